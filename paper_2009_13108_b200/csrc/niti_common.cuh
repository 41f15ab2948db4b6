// Shared declarations of the NITI sm_100a library (internal; the public boundary is include/niti.h).
#pragma once
#include <cuda_runtime.h>
#include <cuda.h>
#include <stdint.h>
#include <stdio.h>
#include <string.h>

#include "../../include/niti.h"

struct niti_ctx {
  int device;
  int sm_count;
  int engine;               // niti_set_engine: 0 auto, 1 CUDA-core kernels only, 2 single-CTA tensor-core kernel,
                            // 3 paired-CTA only, 4 two-pass (int32 spill) epilogue, 5 no resident-weights mode
  uint32_t *d_status;       // device status word (+ counter of recomputations)
  int32_t *d_spec_tab;      // NITI_SPEC_SLOTS x {tag, error}: per call site, by how many bits the sample-based
                            // estimate of the speculative epilogue missed the true bit-width last time
  uint64_t launches;
  uint64_t tc_launches;     // launches of the tensor-core matrix-multiply kernels (two multiplies in one count as two)
  uint64_t tc2_launches;    // of those, launches of the paired-CTA (cta_group::2) variant
  uint64_t res_launches;    // and launches of the generic loops with all of B resident
  char err[256];
  // optional timing of the tensor-core kernel: event pairs recorded around each launch
  int profile_on;
  int prof_used;
  cudaEvent_t *prof_ev;     // 2 * NITI_PROF_MAX events
  double *prof_ops;         // algorithmic int8 operations (2*M*N*K) of each recorded launch
  // cuTensorMapEncodeTiled, fetched through the runtime so that libcuda is not a link dependency
  void *encode_tiled;
  void *encode_im2col;      // cuTensorMapEncodeIm2col
  // data-parallel training (niti_set_reduce_hook): called where a tensor-wide quantity has to be
  // combined over the ranks before the rounding may use it
  niti_reduce_fn reduce_fn;
  void *reduce_user;
  // niti_set_tap_cache: caller-owned buffer that keeps the gathered taps of a few-channel convolution
  // between its forward call and its weight-gradient call, and what it currently holds
  int8_t *tap_buf;
  size_t tap_bytes;
  const void *tap_x;
  int tap_dims[9];          // B, H, W, Cin, R, S, pad, stride, valid
  // niti_begin_step: workspace whose headers were cleared in one go, and how many of them are used up
  void *step_ws;
  int step_slot;
  unsigned long long step_capture;  // the capture that niti_begin_step was part of (0: none)
  struct WsHeader *dirty_hdr;   // header of the call being enqueued that has not been cleared yet, or null
  // niti_own_workspace: calls alternate between two headers of this workspace, each clearing the other one's
  void *own_ws;
  int own_next;             // which of the two the next call takes
  int own_clean;            // that one is zero by the time the next call runs
  int own_taken;            // the call being enqueued has taken it
  int dp_rank, dp_world;    // niti_set_dp_shard: > 1 ranks = weight gradients are reduce-scattered, rounded per
                            // shard and all-gathered as int8 (5 bytes per weight on the wire instead of 8)
  // per-device facts of the tensor-core kernel, indexed by CTAs per tile (1 or 2): co-resident CTAs /
  // CTA pairs (0 = not asked yet) and the dynamic shared-memory limit already set on the kernel
  int tc_units[3];
  size_t tc_attr_smem[13];  // CTAs + 2 * mode + 6 * one of the instance
  // the device's opt-in limit of dynamic shared memory per CTA.  The limit set on a kernel belongs to the
  // device, not to a context: every context therefore sets this same value (a context that set only what it
  // needed would lower the limit under another context of the process)
  size_t smem_optin;
  int small_ready;          // attributes of the small-multiply kernel are set
  unsigned patience;        // cycles that the blocks of a launch wait for each other (NITI_PATIENCE; 0: test switch)
};



#define NITI_PROF_MAX 8192
#define NITI_SPEC_SLOTS 4096
// Every workspace starts with NITI_HDR_SLOTS headers of NITI_HDR_SLOT_BYTES each (reduction scalars, the
// words of the speculative agreement, split maxima).  A call needs a zeroed header.  Without further
// notice it clears and uses the last one.  After niti_begin_step() has cleared all of them with one
// launch, the following calls on that workspace take one header each, in order, without clearing (a
// header cleared per call costs a launch of about 1 us in front of every multiply of a step).
#define NITI_HDR_SLOTS 64
#define NITI_HDR_OWN 61                       // this one and the next: see niti_take_header
#define NITI_HDR_SLOT_BYTES 4096
#define NITI_WS_HEADER (NITI_HDR_SLOTS * NITI_HDR_SLOT_BYTES)   // bytes in front of the accumulator scratch
// A contraction that is split over CTAs adds int32 partial sums; split s records the largest magnitude
// among its partial sums in split_max[s] (unsigned words from byte NITI_SPLIT_MAX_OFF of the header).
// The sum of those maxima bounds every accumulator of the tensor: when it reaches 2^31 the int32
// contract of Section 3.2 can no longer be vouched for and NITI_DEV_ACC_RANGE is raised.  Every split
// covers at most NITI_SPLIT_MAX_K contraction elements, so a partial sum itself cannot wrap.
#define NITI_SPLIT_MAX_OFF 256
#define NITI_MAX_SPLITS 960
#define NITI_SPLIT_MAX_K 131072

// Scalars at the start of a workspace.
struct WsHeader {
  unsigned int maxabs32;            // a value with the bit length of max |acc| (a max, or an OR of magnitudes)
  unsigned int arrived;             // agreement of a launch's blocks: low half blocks that have come, high half that left
  unsigned long long maxabs64;      // same for the 64-bit loss accumulators
  unsigned int spec_mask;           // bit b: a CTA of a speculative launch has rounded with bit-width b
  unsigned int hits;                // integer cross-entropy: rows whose first arg-max is the label
};
static_assert(sizeof(WsHeader) == 24, "workspace header layout");
static_assert(NITI_SPLIT_MAX_OFF + 4 * NITI_MAX_SPLITS <= NITI_HDR_SLOT_BYTES, "split maxima fit the header");
__host__ __device__ __forceinline__ unsigned int *niti_split_max(WsHeader *hdr) {
  return reinterpret_cast<unsigned int *>(reinterpret_cast<char *>(hdr) + NITI_SPLIT_MAX_OFF);
}

#define NITI_CUDA_TRY(ctx, expr)                                                        \
  do {                                                                                  \
    cudaError_t e__ = (expr);                                                           \
    if (e__ != cudaSuccess) {                                                           \
      snprintf((ctx)->err, sizeof((ctx)->err), "%s failed: %s (%s:%d)", #expr,          \
               cudaGetErrorString(e__), __FILE__, __LINE__);                            \
      return NITI_ERR_CUDA;                                                             \
    }                                                                                   \
  } while (0)

// Launches are programmatic dependents of the kernel before them in the stream: blocks may become resident while that one
// drains, and its launch latency and set-up overlap its tail.  Every kernel of the library calls niti_enter() before it
// touches global memory: it waits until the kernels before it have completed and are visible, and only then lets the next
// one be scheduled, so that at most two kernels of a stream are resident and the order of all accesses is the stream's.
// The pointers that a kernel reads through go through an empty assembler statement, because loads through restricted
// pointers to constant data may otherwise be moved up across the wait.  Measured against plain
// launches and memsets: classifier head of 4096 x 1000 x 512 (9 launches) 83.7 -> 70.2 us, forward, error and gradient of a
// 56 x 56 layer 90 -> 82 us, one 256^3 multiply 9.1 -> 8.0 us, an eager LeNet step 204 -> 191 us; inside a graph 1 - 3 %.
template <typename... P>
__device__ __forceinline__ void niti_enter(P &...p) {
  asm volatile("griddepcontrol.wait;" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  (void)(int[]){0, ([&] { asm volatile("" : "+l"(p)::"memory"); }(), 0)...};
}
template <typename... K, typename... A>
static inline cudaError_t niti_launch(cudaStream_t st, dim3 grid, dim3 block, size_t smem, void (*kernel)(K...), A... args) {
  cudaLaunchConfig_t cfg;
  memset(&cfg, 0, sizeof(cfg));
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kernel, args...);
}

// Zeroes `bytes` (a multiple of 4) from a 16-byte boundary with a kernel: unlike a memset it takes part in the overlap.
int niti_memset0(niti_ctx *ctx, cudaStream_t st, void *p, size_t bytes);
static inline WsHeader *niti_own_header(void *ws, int which) {
  return reinterpret_cast<WsHeader *>(reinterpret_cast<char *>(ws) + (size_t)NITI_HDR_SLOT_BYTES * (NITI_HDR_OWN + which));
}
// The capture that a stream is part of; 0: none, NITI_CAPTURE_UNKNOWN: the stream cannot say (another one is being captured).
#define NITI_CAPTURE_UNKNOWN (~0ull)
static inline unsigned long long niti_capture_id(cudaStream_t st) {
  cudaStreamCaptureStatus status = cudaStreamCaptureStatusNone;
  unsigned long long id = 0;
  if (cudaStreamGetCaptureInfo(st, &status, &id) != cudaSuccess) {
    (void)cudaGetLastError();
    return NITI_CAPTURE_UNKNOWN;
  }
  return status == cudaStreamCaptureStatusNone ? 0ull : status == cudaStreamCaptureStatusActive ? id : NITI_CAPTURE_UNKNOWN;
}
// A header for the call that is being enqueued: the next unused one of a workspace prepared by niti_begin_step()
// (zeroed already, if the call and niti_begin_step are enqueued alike: a begin that is being captured has cleared nothing yet,
// and one in front of a capture does not repeat with the replays); in a workspace that is this context's own one of two that
// the calls use in turn, the kernel of each clearing the other one for the next (a launch of its own for that took 1.2 us of
// each call: one 256^3 multiply 7.9 -> 6.3 us, forward, error and gradient of a 56 x 56 layer 73.2 -> 71.0 us); else the last
// one, which niti_clear() has to clear before the call's first kernel.  The last one ends where the accumulators begin, so
// that a split contraction clears both with one launch.  A call that is being captured takes the last one too: its replays
// do not alternate.  (So do calls past the 64th of a step, and those without patience, whose test looks there.)
static inline WsHeader *niti_take_header(niti_ctx *ctx, cudaStream_t st, void *ws) {
  char *base = reinterpret_cast<char *>(ws);
  ctx->own_taken = 0;
  ctx->dirty_hdr = nullptr;
  const bool step = ws == ctx->step_ws;
  if (step || ws == ctx->own_ws) {
    const unsigned long long capture = niti_capture_id(st);
    const bool in_step = step && capture == ctx->step_capture && capture != NITI_CAPTURE_UNKNOWN;
    if (in_step && ctx->step_slot < NITI_HDR_SLOTS) {
      if (ws == ctx->own_ws && ctx->step_slot >= NITI_HDR_OWN) {
        ctx->own_clean = 0;
        if (capture) ctx->own_ws = nullptr;                  // (the replays will use them, too)
      }
      return reinterpret_cast<WsHeader *>(base + (size_t)NITI_HDR_SLOT_BYTES * ctx->step_slot++);
    }
    if (ws == ctx->own_ws && !in_step && capture == 0 && ctx->patience) {
      if (!ctx->own_clean) ctx->own_clean = niti_memset0(ctx, st, niti_own_header(ws, 0), 2 * NITI_HDR_SLOT_BYTES) == NITI_OK;
      if (ctx->own_clean) {
        ctx->own_taken = 1;
        return niti_own_header(ws, ctx->own_next);
      }
    }
  }
  ctx->dirty_hdr = reinterpret_cast<WsHeader *>(base + (size_t)NITI_HDR_SLOT_BYTES * (NITI_HDR_SLOTS - 1));
  return ctx->dirty_hdr;
}
// Clears the header taken last if that is still to be done, and the accumulators (acc may be null).  *next: a header that the
// call's first kernel has to zero (null: none), followed by niti_header_passed_on(); callers without such a kernel pass null.
static inline int niti_clear(niti_ctx *ctx, cudaStream_t st, int32_t *acc = nullptr, size_t acc_bytes = 0, WsHeader **next = nullptr) {
  char *hdr = reinterpret_cast<char *>(ctx->dirty_hdr);
  ctx->dirty_hdr = nullptr;
  if (hdr && acc && hdr + NITI_HDR_SLOT_BYTES == reinterpret_cast<char *>(acc))
    return niti_memset0(ctx, st, hdr, NITI_HDR_SLOT_BYTES + acc_bytes);
  int rc = NITI_OK;
  if (hdr) rc = niti_memset0(ctx, st, hdr, NITI_HDR_SLOT_BYTES);
  if (rc == NITI_OK && acc) rc = niti_memset0(ctx, st, acc, acc_bytes);
  if (next) *next = nullptr;
  if (rc == NITI_OK && ctx->own_taken) {
    ctx->own_taken = 0;
    ctx->own_next ^= 1;
    ctx->own_clean = 0;                              // (until something that zeroes the other header is enqueued)
    WsHeader *other = niti_own_header(ctx->own_ws, ctx->own_next);
    if (next) *next = other;
    else ctx->own_clean = (rc = niti_memset0(ctx, st, other, NITI_HDR_SLOT_BYTES)) == NITI_OK;
  }
  return rc;
}
static inline void niti_header_passed_on(niti_ctx *ctx, const WsHeader *next) {
  if (next) ctx->own_clean = 1;
}
// by one warp
__device__ __forceinline__ void niti_zero_header(WsHeader *hdr, int lane) {
#pragma unroll
  for (int i = 0; i < NITI_HDR_SLOT_BYTES / 512; ++i) reinterpret_cast<int4 *>(hdr)[32 * i + lane] = make_int4(0, 0, 0, 0);
}

static inline int niti_fail(niti_ctx *ctx, int code, const char *msg) {
  if (ctx) snprintf(ctx->err, sizeof(ctx->err), "%s", msg);
  return code;
}

// Runs the caller's reduction over the ranks on a device buffer, ordered on the stream.
static inline int niti_reduce(niti_ctx *ctx, cudaStream_t st, void *dev_ptr, long long count, int kind) {
  if (!ctx->reduce_fn) return NITI_OK;
  if (ctx->reduce_fn(ctx->reduce_user, (void *)st, dev_ptr, (int64_t)count, kind) != 0)
    return niti_fail(ctx, NITI_ERR_ARG, "the reduction hook reported a failure");
  return NITI_OK;
}
// (weight gradients contract over the batch: under data parallelism their int32 sums are added
// over the ranks; every other multiply only shares its max magnitude)
static inline bool niti_is_wgrad(int kind) { return kind == 2 || kind == 5; }   // GK_FC_WGRAD, GK_CONV_WGRAD

// ---- rounding arithmetic (Algorithm 3 and round-to-nearest), on the magnitude ----------------
template <typename U>
__device__ __forceinline__ U niti_round_mag(U m, int bp, U qmax, int round_mode) {
  U q = m >> bp;
  U f = m & ((U(1) << bp) - 1);
  if (round_mode == NITI_ROUND_PSR) {
    f >>= (bp & 1);               // odd binary point: the lowest discarded bit is dropped
    int h = bp >> 1;              // width of each half
    U top = f >> h;
    U bot = f & ((U(1) << h) - 1);
    q += (top > bot) ? 1 : 0;
  } else {
    q += (bp > 0 && (f >> (bp - 1))) ? 1 : 0;
  }
  return q > qmax ? qmax : q;
}

__device__ __forceinline__ int niti_round_i32(int x, int bp, unsigned qmax, int round_mode) {
  unsigned m = x < 0 ? 0u - (unsigned)x : (unsigned)x;
  int q = (int)niti_round_mag<unsigned>(m, bp, qmax, round_mode);
  return x < 0 ? -q : q;
}

__device__ __forceinline__ int niti_bitlen32(unsigned v) { return 32 - __clz(v); }

// Four bytes from p, those from the n-th on zero; reads only aligned words that hold at least one wanted byte.
__device__ __forceinline__ unsigned niti_load_bytes4(const int8_t *p, int n) {
  if (n <= 0) return 0u;
  const unsigned mis = (unsigned)(uintptr_t)p & 3u;
  const unsigned *q = reinterpret_cast<const unsigned *>((uintptr_t)p - mis);
  const unsigned lo = q[0];
  const unsigned hi = mis + (unsigned)(n < 4 ? n : 4) > 4u ? q[1] : 0u;
  const unsigned v = __funnelshift_r(lo, hi, 8u * mis);
  return n >= 4 ? v : v & (0xffffffffu >> (32 - 8 * n));
}

// Agreement of the blocks of one launch on the bit-width of a tensor of which every block holds a share: the largest bit
// length over n blocks (at most NITI_AGREE_MAX), plus one, for one converged warp of every block; 0: the block ran out of
// patience and has to leave.  Words [0, n) of the area take what the blocks post.  Up to NITI_AGREE_DIRECT CTAs all poll all
// words; with more, the first CTA alone does and answers into a mailbox of 16 bytes per CTA that only that CTA polls, because
// the reads of a few L2 lines by everybody delay the posts (3100 cycles for 64 CTAs, 6000 - 8000 for 128; one call with 98
// CTAs 12.0 -> 10.5 us, with 64 14.1 -> 13.0 us, with 144 16.0 -> 13.7 us; with 16 6.9 us directly, 7.5 us through
// mailboxes).  `extra` more words in front of the area have to be posted first.
//
// Nothing promises that all blocks of a launch are on the GPU at the same time: launches of two streams can each hold a part
// of the SMs.  So no block waits until all have come.  Out of patience, it leaves its sums in memory, marks its post, counts
// itself as left and exits, which frees its SM for the blocks that are still to come (niti_finish_left).  Arrivals and
// departures are counted in one word, whose order decides who finishes the share of a block that left: the block itself
// when all had arrived by then, else the block that arrived last.  (A cooperative launch would promise residency; it cost
// every launch of a call-by-call program 1.3 us of host time: head of 4096 x 1000 x 512 66.1 -> 72.9 us, eager CNN step of
// 37 launches 169 -> 187 us, one 256^3 multiply 7.8 -> 8.5 us, a captured MLP step 43.2 -> 45.0 us.)
#define NITI_AGREE_MAX 160
#define NITI_AGREE_DIRECT 48
#define NITI_AGREE_WORDS (5 * NITI_AGREE_MAX)      // posts, then mailboxes
#define NITI_LEFT 0x10000u                         // mark in a post: its block left its share in memory
#define NITI_PATIENCE (1u << 19)                   // about 0.3 ms; the blocks of an undisturbed launch post within a few us
__device__ __forceinline__ unsigned niti_agree_bits(unsigned *posts, unsigned *mail, int bits, int cta, int n, int extra, int lane,
                                                    unsigned patience) {
  if (lane == 0) *(volatile unsigned *)(posts + cta) = (unsigned)bits + 1u;
  if (patience == 0u && (cta & 1)) return 0u;      // (test switch: every other block leaves, whoever has come)
  const long long t0 = clock64();
  auto late = [&]() { return __any_sync(0xffffffffu, clock64() - t0 > (long long)patience) != 0; };
  if (cta == 0 || n <= NITI_AGREE_DIRECT) {
    unsigned m;
    while (true) {
      bool seen = true;
      m = 0;
      unsigned w[5];
#pragma unroll
      for (int u = 0; u < 5; ++u) {
        const int i = 32 * u + lane - extra;
        w[u] = i < n ? *(volatile unsigned *)(posts + i) : 1u;
      }
#pragma unroll
      for (int u = 0; u < 5; ++u) {
        const int i = 32 * u + lane - extra;
        seen = seen && w[u] != 0;
        if (i >= 0 && i < n) m = max(m, w[u] & (NITI_LEFT - 1u));
      }
      if (__all_sync(0xffffffffu, seen)) break;
      if (late()) return 0u;
    }
    m = __reduce_max_sync(0xffffffffu, m);
    if (n > NITI_AGREE_DIRECT)
      for (int i = lane; i < n; i += 32) *(volatile unsigned *)(mail + 4 * i) = m;
    return m;
  }
  unsigned m = 0;
  while (true) {
    if (lane == 0) m = *(volatile unsigned *)(mail + 4 * cta);
    m = __shfl_sync(0xffffffffu, m, 0);
    if (m) return m;
    if (late()) return 0u;
  }
}
// The same maximum when all n blocks have arrived: each of them posts without waiting for another.
__device__ __forceinline__ unsigned niti_posted_bits(unsigned *posts, int n, uint32_t *status) {
  unsigned m = 0;
  const long long t0 = clock64();
  for (int i = (int)(threadIdx.x & 31); i < n; i += 32) {
    unsigned w;
    while (!(w = *(volatile unsigned *)(posts + i)))
      if (clock64() - t0 > 2000000000LL) {
        atomicOr(status, NITI_DEV_TIMEOUT);
        break;
      }
    m = max(m, w & (NITI_LEFT - 1u));
  }
  __syncwarp();
  return __reduce_max_sync(0xffffffffu, m);
}
// At the start of every block of such a launch, by one thread, for niti_finish_left.
__device__ __forceinline__ unsigned niti_arrive(WsHeader *hdr) { return atomicAdd(&hdr->arrived, 1u); }
// The end of every block of such a launch, by all its threads: after its own output is stored, or (`left`) after its share
// is in memory.  `ticket`: from niti_arrive, `posts`: of the whole grid.  finish(j) completes the share of block j, which
// left, and is called for every such block by exactly one block.
template <typename Finish>
__device__ __forceinline__ void niti_finish_left(WsHeader *hdr, unsigned *posts, bool left, unsigned ticket, Finish finish) {
  const unsigned n = gridDim.x;
  __shared__ unsigned claimed;
  bool look = (ticket & 0xffffu) == n - 1u && (ticket >> 16) != 0;              // the last to arrive, and some had left
  if (left) {
    __threadfence();                               // (each thread's part of the share)
    __syncthreads();
    if (threadIdx.x == 0) {
      atomicOr(posts + blockIdx.x, NITI_LEFT);
      __threadfence();
      claimed = (atomicAdd(&hdr->arrived, 0x10000u) & 0xffffu) == n ? 1u : 0u;  // (nobody else looks at this block then)
    }
    __syncthreads();
    look = look || claimed != 0;
  }
  if (!look) return;
  __threadfence();
  for (unsigned j = 0; j < n; ++j) {
    __syncthreads();
    if (threadIdx.x == 0) {
      claimed = (*(volatile unsigned *)(posts + j) & NITI_LEFT) && (atomicAnd(posts + j, ~NITI_LEFT) & NITI_LEFT) ? 1u : 0u;
      __threadfence();
    }
    __syncthreads();
    if (claimed) finish((int)j);
  }
}

// ---- internal launchers (defined across the .cu files) ----------------------------------------
// Shape of one matrix multiply D[m][n] = sum_k A(m,k) * B(n,k) with implicit operand addressing.
enum NitiGemmKind {
  GK_FC_FWD = 0,   // A = a[M][K],        B = w[N][K]
  GK_FC_DGRAD,     // A = e[M][N],        B(k', n) = w[n][k']
  GK_FC_WGRAD,     // A(n, m) = e[m][n],  B(k', m) = a[m][k']
  GK_CONV_FWD,     // A(pix, (r,s,ci)) = x shifted, B = w[co][(r,s,ci)]
  GK_CONV_DGRAD,   // A(pix, (r,s,co)) = e shifted, B(ci, (r,s,co)) = w[co][r][s][ci]
  GK_CONV_WGRAD    // A(co, pix) = e[pix][co],      B((r,s,ci), pix) = x shifted
};
static_assert(GK_FC_WGRAD == 2 && GK_CONV_WGRAD == 5, "niti_is_wgrad");

struct GemmProblem {
  int kind;
  const int8_t *p0;  // first operand  (a / e / x)
  const int8_t *p1;  // second operand (w / a / e)
  // fully connected: M, N, K of the layer.  convolution: B,H,W (input), Ho,Wo (output), Ci, Co, R, S, pad, stride
  int M, N, K;
  int B, H, W, Ho, Wo, Ci, Co, R, S, pad, stride;
  // the matrix multiply actually run
  long long gm, gn, gk;
  // Operands as the tensor-core engine copies them, when the caller's rows are no multiple of 16 bytes: copies
  // of p0 / p1 with padded rows (null: the operand itself) and their row pitches in bytes (0: dense).  A row is
  // a row of a matrix, a pixel's channels, or a tap's input channels (convolution weights).
  const int8_t *q0, *q1;
  long long ld0, ld1;
  // windows of a few-channel convolution (0: none): channels of a window, byte distance of neighbouring windows and
  // of image rows in the widened input; W and S then count windows and tap rows' windows (Wo and 1), and only rows
  // have a stride and padding
  int win_chans, win_sw, win_sh;
  int in_place;             // an output is in the storage of an operand or of the gate (set and read by niti_tc_gemm)
};

// shard_ok: the caller rounds only this rank's shard afterwards (niti_dp_shard) and all-gathers the result
int niti_reduce_after_gemm(niti_ctx *ctx, cudaStream_t st, int kind, int32_t *acc, long long n, WsHeader *hdr,
                           bool shard_ok = false);
// Sharding of a weight-gradient tensor of n elements over the data-parallel ranks: `main` elements are
// split evenly (every shard a multiple of 16 elements, so that vector accesses stay aligned), the
// remaining `n - main` are combined with an all-reduce and handled by every rank.
struct NitiDpShard { long long main, shard, off; };
static inline NitiDpShard niti_dp_shard(const niti_ctx *ctx, long long n) {
  NitiDpShard s;
  const long long unit = 16LL * ctx->dp_world;
  s.main = n / unit * unit;
  s.shard = s.main / ctx->dp_world;
  s.off = s.shard * ctx->dp_rank;
  return s;
}
static inline bool niti_dp_sharded(const niti_ctx *ctx, int kind) {
  return ctx->reduce_fn && ctx->dp_world > 1 && (kind == 2 || kind == 5);   // weight gradients only
}
// max |acc| into hdr->maxabs32; splits > 1: also adds up the split maxima of the header and raises
// NITI_DEV_ACC_RANGE when an accumulator may have left the int32 range
int niti_launch_maxabs(niti_ctx *ctx, cudaStream_t st, const int32_t *acc, long long n, WsHeader *hdr, int splits = 0);
// Plain CUDA-core engine: writes int32 accumulators to acc[gm][gn] and max|acc| to hdr->maxabs32.
int niti_simt_gemm(niti_ctx *ctx, cudaStream_t st, const GemmProblem &p, int32_t *acc, WsHeader *hdr);
// What follows the multiply: rounding target and the scalars of Algorithm 2.
struct RoundSpec {
  int8_t *out;
  const int8_t *mask;      // optional ReLU mask source (zero the output where mask <= 0)
  int mbits, round_mode, relu;
  const int32_t *s_a, *s_w;
  int32_t *s_out, *b_out;
  int8_t *pool_out;        // optional (may be null): 2 x 2 max-pool of `out`, forward convolutions with ReLU
  // (out may be null: the caller wants the int32 accumulators and rounds them itself)
  int8_t *update_w;        // optional (may be null): weight gradients; the caller will subtract `out` from these weights
};
// Tensor-core engine (tcgen05); returns NITI_ERR_SHAPE if the shape is not eligible.  *fused is set
// when the kernel also did the bit-width / shift / round / store (nothing is left to do); otherwise
// acc holds the int32 accumulators and hdr->maxabs32 their max magnitude.
// *pooled (may be null) is set when the kernel's epilogue also wrote r.pool_out.
// *updated (may be null) is set when the epilogue subtracted the rounded gradient from r.update_w itself
// (`out` is then not written).
int niti_tc_gemm(niti_ctx *ctx, cudaStream_t st, const GemmProblem &p, const RoundSpec &r, int32_t *acc,
                 WsHeader *hdr, bool *fused, bool *pooled = nullptr, bool shard_ok = false, bool *updated = nullptr);

// Small fully connected multiplies, one launch for one (g2 == null) or both multiplies of a backward call;
// NITI_ERR_SHAPE when the problem is not small (nothing was enqueued).
#define NITI_SMALL_MACS 200.0e6
#define NITI_SMALL_NARROW 4                        // times that for layers of fewer than 32 outputs, backward
int niti_small_gemm(niti_ctx *ctx, cudaStream_t st, void *ws, const GemmProblem &g, const RoundSpec &r,
                    const GemmProblem *g2, const RoundSpec *r2);

// Epilogue pass: b from hdr->maxabs32, bp = max(0, b - mbits), out = Round(acc) with optional ReLU
// and optional mask; s_out = s_a + s_w + bp if s_out != NULL; b_out = b if != NULL.
int niti_launch_round(niti_ctx *ctx, cudaStream_t st, const int32_t *acc, const WsHeader *hdr,
                      int8_t *out, long long n, int mbits, int round_mode, int relu,
                      const int8_t *mask, const int32_t *s_a, const int32_t *s_w, int32_t *s_out,
                      int32_t *b_out, int8_t *upd_w = nullptr);
