// C-ABI entry points of the NITI library: argument checks, engine selection, and the
// accumulate -> bit-width -> shift-and-round sequence of Algorithm 1 for each layer op.
#include "niti_common.cuh"

int niti_launch_im2col32(niti_ctx *ctx, cudaStream_t st, const int8_t *x, int8_t *xcol, int B, int H, int W,
                         int Ci, int R, int S, int pad, int stride, int Ho, int Wo);
int niti_launch_widen(niti_ctx *ctx, cudaStream_t st, const int8_t *x, int8_t *xw, int rows, int W, int Ci, int Cp, int pad,
                      int row_bytes, const int8_t *w, int8_t *ww, int wrows, int S, int pitch);
int niti_launch_pad_pitch(niti_ctx *ctx, cudaStream_t st, const int8_t *src, int8_t *dst, long long rows, int n, int pitch);
int niti_launch_round_compact(niti_ctx *ctx, cudaStream_t st, const int32_t *acc, const WsHeader *hdr, int8_t *out,
                              int rows, int k, int pitch, int rowk, int rpitch, int Ci, int Cp, int mbits, int round_mode,
                              int32_t *b_out, int8_t *upd_w);

static inline size_t round_up(size_t v, size_t a) { return (v + a - 1) / a * a; }

// Few-channel convolutions (first layers: Cin = 1 or 3, no TMA view of the NHWC tensor), forward and weight
// gradient.  With at most 32 taps the taps of every output pixel are gathered into one 32-byte row and the layer
// runs as a plain K = 32 matrix multiply.
static inline bool few_channel_conv(int Ci, int R, int S) { return R * S * Ci <= 32 && (Ci % 16) != 0; }

// A forward pass or weight gradient with a stride above 8 has no operand copies on the tensor-core engine (the traversal
// stride of a copy ends there): the CUDA-core engine reads the caller's tensors, nothing is widened or padded for it.
static inline bool copies_refused(const GemmProblem &p) {
  return (p.kind == GK_CONV_FWD || p.kind == GK_CONV_WGRAD) && p.stride > 8;
}

// With more taps nothing is gathered: a tap row of a window is S * Ci contiguous bytes of an image row.  Pixels are
// widened to Cp bytes (4, 8 or 16: stride * Cp has to be a multiple of the 16 bytes that TMA strides are made of)
// and image rows get their zero padding, and then the layer is a convolution with R x 1 taps over Wo "pixels" per
// row that lie stride * Cp bytes apart and have S * Cp channels: windows that overlap in memory.
//
// The workspace query and the calls decide by the same rules here: what a call copies is what the query has room for.
struct WindowGeometry {
  int Cp;                  // bytes per widened pixel, 0: the layer is not run this way
  int row_bytes;           // of a widened image row
  int chans, pitch;        // channels of a window (S * Cp), and rounded up to 16: pitch of a tap row of weights
  size_t x_bytes, w_bytes, acc_bytes;
};
static WindowGeometry window_geometry(const GemmProblem &p) {
  WindowGeometry g;
  memset(&g, 0, sizeof(g));
  if (p.Ci >= 16 || few_channel_conv(p.Ci, p.R, p.S) || p.kind == GK_CONV_DGRAD || copies_refused(p)) return g;
  // (the box of base pixels that an im2col copy walks starts and ends within 128 rows of the image's)
  if (p.pad > 127 || p.R - 1 - p.pad > 128) return g;
  int cp = 4;
  while (cp < p.Ci || (p.stride * cp) % 16 != 0) cp *= 2;
  if (cp > 16) return g;
  const long long row_bytes = (((p.Wo - 1LL) * p.stride + p.S) * cp + 15) / 16 * 16;
  if ((long long)p.B * p.H * (row_bytes / 16) >= (1LL << 31)) return g;       // (the widening kernel counts in 32 bits)
  g.Cp = cp;
  g.row_bytes = (int)row_bytes;
  g.chans = p.S * cp;
  g.pitch = (g.chans + 15) / 16 * 16;
  g.x_bytes = round_up((size_t)p.B * p.H * g.row_bytes, 256);
  g.w_bytes = round_up((size_t)p.Co * p.R * g.pitch, 256);
  g.acc_bytes = round_up((size_t)p.Co * p.R * g.pitch * 4, 256);
  return g;
}
// The problem as the tensor-core engine sees it.
static GemmProblem window_problem(const GemmProblem &p, const WindowGeometry &g, const int8_t *xw) {
  GemmProblem q = p;
  q.Ci = g.pitch;
  q.W = p.Wo; q.S = 1;
  q.win_chans = g.chans;
  q.win_sw = p.stride * g.Cp; q.win_sh = g.row_bytes;
  if (p.kind == GK_CONV_FWD) { q.gk = (long long)p.R * g.pitch; q.q0 = xw; }
  else { q.gn = (long long)p.R * g.pitch; q.q1 = xw; }
  return q;
}

// An operand of a multiply as rows of `width` bytes; TMA needs row pitches that are multiples of 16, so other
// widths are copied once per call into padded rows (q0 / q1 of the problem).
struct OperandRows { long long rows; int width; };
static OperandRows operand_rows(const GemmProblem &p, int which) {
  switch (p.kind) {
    case GK_FC_FWD: return which == 0 ? OperandRows{p.M, p.K} : OperandRows{p.N, p.K};
    case GK_FC_DGRAD: return which == 0 ? OperandRows{p.M, p.N} : OperandRows{p.N, p.K};
    case GK_FC_WGRAD: return which == 0 ? OperandRows{p.M, p.N} : OperandRows{p.M, p.K};
    default: break;
  }
  const OperandRows x = {(long long)p.B * p.H * p.W, p.Ci}, e = {(long long)p.B * p.Ho * p.Wo, p.Co};
  const OperandRows w = {(long long)p.Co * p.R * p.S, p.Ci};
  if (p.kind == GK_CONV_FWD) return which == 0 ? x : w;
  if (p.kind == GK_CONV_DGRAD) return which == 0 ? e : w;
  return which == 0 ? e : x;
}
static inline int pitch16(int width) { return (width + 15) / 16 * 16; }
static size_t pad_bytes(const GemmProblem &p, int which) {
  const OperandRows o = operand_rows(p, which);
  return o.width % 16 == 0 ? 0 : round_up((size_t)o.rows * pitch16(o.width), 256);
}
static size_t pad_bytes(const GemmProblem &p) { return pad_bytes(p, 0) + pad_bytes(p, 1); }
// Copies what needs padding (and is not padded yet) into `mem` (pad_bytes(p) bytes); `end`: end of the workspace.
static int pad_operands(niti_ctx *ctx, cudaStream_t st, GemmProblem &p, char *mem, const char *end) {
  for (int which = 0; which < 2; ++which) {
    const size_t bytes = pad_bytes(p, which);
    const int8_t *&q = which == 0 ? p.q0 : p.q1;
    if (bytes && !q) {
      const OperandRows o = operand_rows(p, which);
      if (mem + bytes > end) return niti_fail(ctx, NITI_ERR_WORKSPACE, "the workspace has no room for padded operands");
      const int rc = niti_launch_pad_pitch(ctx, st, which == 0 ? p.p0 : p.p1, (int8_t *)mem, o.rows, o.width, pitch16(o.width));
      if (rc != NITI_OK) return rc;
      q = (int8_t *)mem;
      (which == 0 ? p.ld0 : p.ld1) = pitch16(o.width);
    }
    mem += bytes;
  }
  return NITI_OK;
}

extern "C" int niti_create(niti_ctx **out, int device) {
  if (!out) return NITI_ERR_ARG;
  *out = nullptr;
  niti_ctx *ctx = new niti_ctx();
  memset(ctx, 0, sizeof(*ctx));
  ctx->device = device;
  // (single attributes: the full property query takes about 3 ms)
  int major = 0, smem_optin = 0;
  cudaError_t e = cudaSetDevice(device);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&major, cudaDevAttrComputeCapabilityMajor, device);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&ctx->sm_count, cudaDevAttrMultiProcessorCount, device);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&smem_optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, device);
  if (e != cudaSuccess) {
    delete ctx;
    return NITI_ERR_CUDA;
  }
  if (major != 10) {        // the kernels are built for sm_100a only
    delete ctx;
    return NITI_ERR_SHAPE;
  }
  ctx->smem_optin = (size_t)smem_optin;
  ctx->patience = NITI_PATIENCE;
  // one allocation: the status words, then the table of speculative-estimate errors
  const size_t dev_bytes = 256 + sizeof(int32_t) * 2 * NITI_SPEC_SLOTS;
  e = cudaMalloc(&ctx->d_status, dev_bytes);
  if (e == cudaSuccess) e = cudaMemset(ctx->d_status, 0, dev_bytes);
  if (e != cudaSuccess) {
    delete ctx;
    return NITI_ERR_CUDA;
  }
  ctx->d_spec_tab = (int32_t *)((char *)ctx->d_status + 256);
  cudaDriverEntryPointQueryResult qres;
  void *fn = nullptr;
  if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &fn, cudaEnableDefault, &qres) == cudaSuccess &&
      qres == cudaDriverEntryPointSuccess)
    ctx->encode_tiled = fn;
  fn = nullptr;
  if (cudaGetDriverEntryPoint("cuTensorMapEncodeIm2col", &fn, cudaEnableDefault, &qres) == cudaSuccess &&
      qres == cudaDriverEntryPointSuccess)
    ctx->encode_im2col = fn;
  *out = ctx;
  return NITI_OK;
}

extern "C" int niti_destroy(niti_ctx *ctx) {
  if (!ctx) return NITI_ERR_ARG;
  if (ctx->prof_ev) {
    for (int i = 0; i < 2 * NITI_PROF_MAX; ++i) cudaEventDestroy(ctx->prof_ev[i]);
    delete[] ctx->prof_ev;
    delete[] ctx->prof_ops;
  }
  cudaFree(ctx->d_status);
  delete ctx;
  return NITI_OK;
}

extern "C" const char *niti_last_error(niti_ctx *ctx) { return ctx ? ctx->err : "null context"; }

extern "C" int niti_set_engine(niti_ctx *ctx, int engine) {
  if (!ctx) return -1;
  const int old = ctx->patience ? ctx->engine : 6;
  ctx->engine = engine == 6 ? 0 : engine;
  ctx->patience = engine == 6 ? 0u : NITI_PATIENCE;
  return old;
}

extern "C" int niti_set_reduce_hook(niti_ctx *ctx, niti_reduce_fn fn, void *user) {
  if (!ctx) return NITI_ERR_ARG;
  ctx->reduce_fn = fn;
  ctx->reduce_user = fn ? user : nullptr;
  return NITI_OK;
}

extern "C" int niti_begin_step(niti_ctx *ctx, void *stream, void *ws, size_t ws_bytes) {
  if (!ctx) return NITI_ERR_ARG;
  if (!ws) {                                     // forget the prepared workspace: calls clear their header again
    ctx->step_ws = nullptr;
    ctx->step_slot = 0;
    return NITI_OK;
  }
  if (((uintptr_t)ws & 255) || ws_bytes < NITI_WS_HEADER)
    return niti_fail(ctx, NITI_ERR_WORKSPACE, "niti_begin_step: workspace misaligned or too small");
  const int rc = niti_memset0(ctx, (cudaStream_t)stream, ws, NITI_WS_HEADER);
  if (rc != NITI_OK) return rc;
  ctx->step_ws = ws;
  ctx->step_slot = 0;
  ctx->step_capture = niti_capture_id((cudaStream_t)stream);
  if (ws == ctx->own_ws && ctx->step_capture == 0) ctx->own_clean = 1;        // (its two headers are among the cleared ones)
  return NITI_OK;
}

extern "C" int niti_own_workspace(niti_ctx *ctx, void *ws, size_t ws_bytes) {
  if (!ctx) return NITI_ERR_ARG;
  if (ws && (((uintptr_t)ws & 255) || ws_bytes < NITI_WS_HEADER))
    return niti_fail(ctx, NITI_ERR_WORKSPACE, "niti_own_workspace: workspace misaligned or too small");
  ctx->own_ws = ws;
  ctx->own_next = 0;
  ctx->own_clean = 0;
  return NITI_OK;
}

extern "C" int niti_set_tap_cache(niti_ctx *ctx, void *buf, size_t bytes) {
  if (!ctx || (buf && (((uintptr_t)buf & 255) || bytes == 0))) return NITI_ERR_ARG;
  ctx->tap_buf = (int8_t *)buf;
  ctx->tap_bytes = buf ? bytes : 0;
  ctx->tap_x = nullptr;
  ctx->tap_dims[8] = 0;
  return NITI_OK;
}

// Does the tap cache hold the gathered rows of exactly this input tensor and geometry?
static bool tap_cache_hit(const niti_ctx *ctx, const void *x, int B, int H, int W, int Ci, int R, int S, int pad,
                          int stride) {
  const int want[8] = {B, H, W, Ci, R, S, pad, stride};
  if (!ctx->tap_buf || !ctx->tap_dims[8] || ctx->tap_x != x) return false;
  for (int i = 0; i < 8; ++i)
    if (ctx->tap_dims[i] != want[i]) return false;
  return true;
}

extern "C" int niti_set_dp_shard(niti_ctx *ctx, int rank, int world) {
  if (!ctx || world < 1 || rank < 0 || rank >= world) return NITI_ERR_ARG;
  ctx->dp_rank = rank;
  ctx->dp_world = world;
  return NITI_OK;
}

extern "C" uint64_t niti_launch_count(niti_ctx *ctx) { return ctx ? ctx->launches : 0; }
extern "C" uint64_t niti_tc_launch_count(niti_ctx *ctx) { return ctx ? ctx->tc_launches : 0; }
extern "C" uint64_t niti_tc_pair_launch_count(niti_ctx *ctx) { return ctx ? ctx->tc2_launches : 0; }
extern "C" uint64_t niti_tc_resident_launch_count(niti_ctx *ctx) { return ctx ? ctx->res_launches : 0; }

extern "C" int64_t niti_redo_count(niti_ctx *ctx, void *stream) {
  if (!ctx) return -1;
  uint32_t h = 0;
  if (cudaStreamSynchronize((cudaStream_t)stream) != cudaSuccess) return -1;
  if (cudaMemcpy(&h, ctx->d_status + 1, sizeof(h), cudaMemcpyDeviceToHost) != cudaSuccess) return -1;
  return (int64_t)h;
}

int niti_tc_timeout_probe(niti_ctx *ctx, cudaStream_t st);
extern "C" int niti_selftest_timeout(niti_ctx *ctx, void *stream) {
  if (!ctx) return NITI_ERR_ARG;
  return niti_tc_timeout_probe(ctx, (cudaStream_t)stream);
}

extern "C" int niti_profile_enable(niti_ctx *ctx, int on) {
  if (!ctx) return NITI_ERR_ARG;
  if (on && !ctx->prof_ev) {
    ctx->prof_ev = new cudaEvent_t[2 * NITI_PROF_MAX];
    ctx->prof_ops = new double[NITI_PROF_MAX];
    for (int i = 0; i < 2 * NITI_PROF_MAX; ++i) NITI_CUDA_TRY(ctx, cudaEventCreate(&ctx->prof_ev[i]));
  }
  ctx->profile_on = on ? 1 : 0;
  ctx->prof_used = 0;
  return NITI_OK;
}

extern "C" int niti_profile_read_launches(niti_ctx *ctx, double *ms, double *ops, int max_n) {
  if (!ctx || !ms || !ops || max_n < 0) return -1;
  int n = ctx->prof_used < max_n ? ctx->prof_used : max_n;
  for (int i = 0; i < n; ++i) {
    float t = 0;
    if (cudaEventSynchronize(ctx->prof_ev[2 * i + 1]) != cudaSuccess) return -1;
    if (cudaEventElapsedTime(&t, ctx->prof_ev[2 * i], ctx->prof_ev[2 * i + 1]) != cudaSuccess) return -1;
    ms[i] = t;
    ops[i] = ctx->prof_ops[i];
  }
  return n;
}

extern "C" int niti_profile_read(niti_ctx *ctx, double *tc_ms, uint64_t *tc_launches, double *tc_ops) {
  if (!ctx || !tc_ms || !tc_launches || !tc_ops) return NITI_ERR_ARG;
  double ms = 0, ops = 0;
  for (int i = 0; i < ctx->prof_used; ++i) {
    float t = 0;
    NITI_CUDA_TRY(ctx, cudaEventSynchronize(ctx->prof_ev[2 * i + 1]));
    NITI_CUDA_TRY(ctx, cudaEventElapsedTime(&t, ctx->prof_ev[2 * i], ctx->prof_ev[2 * i + 1]));
    ms += t;
    ops += ctx->prof_ops[i];
  }
  *tc_ms = ms;
  *tc_launches = (uint64_t)ctx->prof_used;
  *tc_ops = ops;
  ctx->prof_used = 0;
  return NITI_OK;
}

extern "C" int niti_check(niti_ctx *ctx, void *stream, uint32_t *status) {
  if (!ctx) return NITI_ERR_ARG;
  uint32_t h = 0;
  NITI_CUDA_TRY(ctx, cudaStreamSynchronize((cudaStream_t)stream));
  NITI_CUDA_TRY(ctx, cudaMemcpy(&h, ctx->d_status, sizeof(h), cudaMemcpyDeviceToHost));
  if (h) NITI_CUDA_TRY(ctx, cudaMemset(ctx->d_status, 0, sizeof(h)));
  if (status) *status = h;
  if (h) {
    snprintf(ctx->err, sizeof(ctx->err), "device status word 0x%x", h);
    return NITI_ERR_DEVICE;
  }
  return NITI_OK;
}

static bool fill_conv(GemmProblem &p, int kind, int B, int H, int W, int Ci, int Co, int R, int S,
                      int pad, int stride = 1) {
  p.kind = kind;
  p.B = B; p.H = H; p.W = W; p.Ci = Ci; p.Co = Co; p.R = R; p.S = S; p.pad = pad; p.stride = stride;
  if (stride < 1 || H + 2 * pad < R || W + 2 * pad < S) return false;
  p.Ho = (H + 2 * pad - R) / stride + 1;
  p.Wo = (W + 2 * pad - S) / stride + 1;
  if (p.Ho <= 0 || p.Wo <= 0) return false;
  if (kind == GK_CONV_FWD) { p.gm = (long long)B * p.Ho * p.Wo; p.gn = Co; p.gk = (long long)R * S * Ci; }
  else if (kind == GK_CONV_DGRAD) { p.gm = (long long)B * H * W; p.gn = Ci; p.gk = (long long)R * S * Co; }
  else { p.gm = Co; p.gn = (long long)R * S * Ci; p.gk = (long long)B * p.Ho * p.Wo; }
  return true;
}

// int32 elements of the accumulator scratch of a fully connected backward call: the larger of the weight
// gradient [N][K] and the error [M][K], both where one launch may run both multiplies
static size_t linear_bwd_acc_elems(long long M, long long N, long long K) {
  const size_t a = (size_t)(M * K), b = (size_t)(N * K);
  if ((double)M * N * K <= NITI_SMALL_MACS * NITI_SMALL_NARROW) return a + b;
  return a > b ? a : b;
}

static void fill_fc(GemmProblem &p, int kind, int M, int N, int K) {
  memset(&p, 0, sizeof(p));
  p.kind = kind; p.M = M; p.N = N; p.K = K;
  if (kind == GK_FC_FWD) { p.gm = M; p.gn = N; p.gk = K; }
  else if (kind == GK_FC_DGRAD) { p.gm = M; p.gn = K; p.gk = N; }
  else { p.gm = N; p.gn = K; p.gk = M; }
}

extern "C" size_t niti_workspace_bytes(int op, const int64_t *d, int nd) {
  if (!d) return 0;
  GemmProblem p, p2;
  memset(&p, 0, sizeof(p));
  memset(&p2, 0, sizeof(p2));
  size_t outs = 0, extra = 0;
  switch (op) {
    case NITI_OP_LINEAR_FWD:
      if (nd != 3 || d[0] <= 0 || d[1] <= 0 || d[2] <= 0) return 0;
      fill_fc(p, GK_FC_FWD, (int)d[0], (int)d[1], (int)d[2]);
      outs = (size_t)(d[0] * d[1]);
      extra = pad_bytes(p);
      break;
    case NITI_OP_LINEAR_BWD_UPDATE:
    case NITI_OP_LINEAR_BWD: {
      if (nd != 3 || d[0] <= 0 || d[1] <= 0 || d[2] <= 0) return 0;
      size_t b = (size_t)(d[1] * d[2]);
      outs = linear_bwd_acc_elems(d[0], d[1], d[2]);
      fill_fc(p, GK_FC_DGRAD, (int)d[0], (int)d[1], (int)d[2]);
      fill_fc(p2, GK_FC_WGRAD, (int)d[0], (int)d[1], (int)d[2]);
      extra = pad_bytes(p) + pad_bytes(p2, 1);        // e, w and a with padded rows
      if (op == NITI_OP_LINEAR_BWD_UPDATE) extra = round_up(extra, 256) + round_up(b, 256);    // scratch gradient
      break;
    }
    case NITI_OP_CONV_FWD:
    case NITI_OP_CONV_DGRAD:
    case NITI_OP_CONV_WGRAD_UPDATE:
    case NITI_OP_CONV_WGRAD: {
      if (nd != 8 && nd != 9) return 0;                  // a ninth entry is the stride (default 1)
      for (int i = 0; i < 7; ++i)
        if (d[i] <= 0) return 0;
      const int stride = nd == 9 ? (int)d[8] : 1;
      const bool upd = op == NITI_OP_CONV_WGRAD_UPDATE;
      if (upd) op = NITI_OP_CONV_WGRAD;
      int kind = op == NITI_OP_CONV_FWD ? GK_CONV_FWD : (op == NITI_OP_CONV_DGRAD ? GK_CONV_DGRAD : GK_CONV_WGRAD);
      if (!fill_conv(p, kind, (int)d[0], (int)d[1], (int)d[2], (int)d[3], (int)d[4], (int)d[5], (int)d[6], (int)d[7],
                     stride))
        return 0;
      outs = (size_t)(p.gm * p.gn);
      const WindowGeometry wg = window_geometry(p);
      if (wg.Cp) {
        extra = wg.x_bytes + wg.w_bytes + wg.acc_bytes;
        if (op == NITI_OP_CONV_WGRAD) extra += pad_bytes(p, 0);           // e with padded pixels
      } else if (few_channel_conv((int)d[3], (int)d[5], (int)d[6]) && op != NITI_OP_CONV_DGRAD) {
        const size_t M = (size_t)d[0] * p.Ho * p.Wo;
        extra = round_up(M * 32, 256) + round_up((size_t)d[4] * 32, 256) + round_up((size_t)d[4] * 32 * 4, 256);
        if (op == NITI_OP_CONV_WGRAD) extra += pad_bytes(p, 0);           // e with padded pixels
      } else if (!copies_refused(p)) {
        extra = pad_bytes(p);
      }
      if (upd) extra = round_up(extra, 256) + round_up((size_t)(p.gm * p.gn), 256);             // scratch gradient
      break;
    }
    case NITI_OP_INT_XENT:
      if (nd != 2 || d[0] <= 0 || d[1] <= 0) return 0;
      // two 64-bit scalars per sample
      return NITI_WS_HEADER + round_up((size_t)d[0] * 16, 256);
    default:
      return 0;
  }
  return NITI_WS_HEADER + round_up(outs * 4, 256) + round_up(extra, 256);
}

static inline bool misaligned16(const void *p) { return ((uintptr_t)p & 15) != 0; }

int niti_launch_sgd_update(niti_ctx *ctx, cudaStream_t st, int8_t *w, const int8_t *g, long long n);

// Data parallelism (niti_set_reduce_hook), after a multiply has left its int32 accumulators in acc and
// their max magnitude in the header: a weight gradient is summed over the ranks and its max taken
// again from the sums; any other tensor only shares the max.
int niti_reduce_after_gemm(niti_ctx *ctx, cudaStream_t st, int kind, int32_t *acc, long long n, WsHeader *hdr,
                           bool shard_ok) {
  if (!ctx->reduce_fn) return NITI_OK;
  if (!niti_is_wgrad(kind)) return niti_reduce(ctx, st, &hdr->maxabs32, 1, NITI_REDUCE_MAX_U32);
  if (shard_ok && niti_dp_sharded(ctx, kind)) {
    // Sharded (Section 3.3's update distributed over the ranks): every rank receives the sums of its own
    // shard only (reduce-scatter, 4 bytes per weight on the wire), the few elements that do not divide
    // evenly are all-reduced, each rank takes the max over what it holds and the maxima are combined.
    // The caller then rounds its shard and all-gathers the int8 result (1 byte per weight).
    const NitiDpShard sh = niti_dp_shard(ctx, n);
    int rc = NITI_OK;
    if (sh.main > 0) rc = niti_reduce(ctx, st, acc, sh.main, NITI_REDUCE_SCATTER_SUM_I32);
    if (rc == NITI_OK && n > sh.main) rc = niti_reduce(ctx, st, acc + sh.main, n - sh.main, NITI_REDUCE_SUM_I32);
    if (rc != NITI_OK) return rc;
    NITI_CUDA_TRY(ctx, cudaMemsetAsync(&hdr->maxabs32, 0, sizeof(unsigned int), st));
    ctx->launches++;
    if (sh.shard > 0) rc = niti_launch_maxabs(ctx, st, acc + sh.off, sh.shard, hdr);
    if (rc == NITI_OK && n > sh.main) rc = niti_launch_maxabs(ctx, st, acc + sh.main, n - sh.main, hdr);
    if (rc != NITI_OK) return rc;
    return niti_reduce(ctx, st, &hdr->maxabs32, 1, NITI_REDUCE_MAX_U32);
  }
  int rc = niti_reduce(ctx, st, acc, n, NITI_REDUCE_SUM_I32);
  if (rc != NITI_OK) return rc;
  NITI_CUDA_TRY(ctx, cudaMemsetAsync(&hdr->maxabs32, 0, sizeof(unsigned int), st));
  ctx->launches++;
  return niti_launch_maxabs(ctx, st, acc, n, hdr);
}

// One matrix multiply of Algorithm 1 followed by EffectiveBitwidth + ShiftAndRound.
// update_w != null (weight gradients): the rounded gradient is not returned but subtracted from the
// weights in place.  When the int32 accumulators exist (split contractions) the rounding pass does
// that itself and the int8 gradient is never stored; when the multiply rounds in its own epilogue,
// `out` is a scratch tensor and the plain update kernel follows.
int niti_launch_maxpool2_fwd(niti_ctx *ctx, cudaStream_t st, const int8_t *x, int8_t *y, int B, int H, int W, int C);

// tc_form: the problem in the form the tensor-core engine takes (operands prepared), where that is another one.
// pad_mem: scratch for operands whose rows have to be padded (pad_bytes(p)).  tc_refused: the tensor-core engine has
// refused the problem already (nothing is padded for it).
static int run_gemm_round(niti_ctx *ctx, cudaStream_t st, GemmProblem p, void *ws, size_t ws_bytes,
                          size_t need, char *pad_mem, int8_t *out, int mbits, int round_mode, int relu,
                          const int8_t *mask, const int32_t *s_a, const int32_t *s_w, int32_t *s_out,
                          int32_t *b_out, int8_t *update_w = nullptr, int8_t *pool_out = nullptr,
                          const GemmProblem *tc_form = nullptr, bool tc_refused = false) {
  if (!ws || ((uintptr_t)ws & 255) || ws_bytes < need)
    return niti_fail(ctx, NITI_ERR_WORKSPACE, "workspace missing, misaligned or too small");
  WsHeader *hdr = niti_take_header(ctx, st, ws);
  int32_t *acc = (int32_t *)((char *)ws + NITI_WS_HEADER);
  int rc = NITI_OK;
  const bool narrow = p.kind <= GK_FC_WGRAD && p.N < 32 && p.kind != GK_FC_FWD;       // (the CUDA-core engine's)
  const bool tc = ctx->engine != 1 && !tc_refused && !copies_refused(p);
  if (tc && !narrow && !tc_form) rc = pad_operands(ctx, st, p, pad_mem, (const char *)ws + need);
  if (rc != NITI_OK) return rc;
  rc = NITI_ERR_SHAPE;
  bool fused = false;
  bool pooled = false;
  bool updated = false;
  RoundSpec rs = {out, mask, mbits, round_mode, relu, s_a, s_w, s_out, b_out, pool_out, update_w};
  if (tc) rc = niti_tc_gemm(ctx, st, tc_form ? *tc_form : p, rs, acc, hdr, &fused, &pooled, true, &updated);
  if (rc == NITI_ERR_SHAPE) {
    rc = niti_simt_gemm(ctx, st, p, acc, hdr);
    if (rc == NITI_OK) rc = niti_reduce_after_gemm(ctx, st, p.kind, acc, p.gm * p.gn, hdr, true);
  }
  if (rc != NITI_OK) return rc;
  if (fused) {
    if (update_w && !updated) return niti_launch_sgd_update(ctx, st, update_w, out, p.gm * p.gn);
  } else if (niti_dp_sharded(ctx, p.kind)) {
    // sharded weight gradient: acc holds the sums over the ranks for this rank's shard (and the
    // remainder): round those (into the gradient, or straight into the weights), then every rank
    // collects the other shards' int8 results
    const long long n = p.gm * p.gn;
    const NitiDpShard sh = niti_dp_shard(ctx, n);
    int8_t *dst = update_w ? update_w : out;
    if (sh.shard > 0)
      rc = niti_launch_round(ctx, st, acc + sh.off, hdr, out + sh.off, sh.shard, mbits, round_mode, relu, nullptr,
                             s_a, s_w, s_out, b_out, update_w ? update_w + sh.off : nullptr);
    if (rc == NITI_OK && n > sh.main)
      rc = niti_launch_round(ctx, st, acc + sh.main, hdr, out + sh.main, n - sh.main, mbits, round_mode, relu, nullptr,
                             s_a, s_w, s_out, b_out, update_w ? update_w + sh.main : nullptr);
    if (rc == NITI_OK && sh.main > 0) rc = niti_reduce(ctx, st, dst, sh.main, NITI_ALLGATHER_I8);
    if (rc != NITI_OK) return rc;
  } else {
    rc = niti_launch_round(ctx, st, acc, hdr, out, p.gm * p.gn, mbits, round_mode, relu, mask, s_a, s_w,
                           s_out, b_out, update_w);
    if (rc != NITI_OK) return rc;
  }
  // the pooled copy of a forward convolution, where the multiply's own epilogue did not write it
  if (pool_out && !pooled) return niti_launch_maxpool2_fwd(ctx, st, out, pool_out, p.B, p.Ho, p.Wo, p.Co);
  return NITI_OK;
}

extern "C" int niti_linear_fwd(niti_ctx *ctx, void *stream, const int8_t *a, const int32_t *s_a,
                               const int8_t *w, const int32_t *s_w, int8_t *out, int32_t *s_out,
                               int32_t *b_out, int M, int N, int K, int relu, int round_mode, void *ws,
                               size_t ws_bytes) {
  if (!ctx) return NITI_ERR_ARG;
  if (!a || !w || !out || !s_a || !s_w || M <= 0 || N <= 0 || K <= 0 || (round_mode != 0 && round_mode != 1) ||
      misaligned16(a) || misaligned16(w) || misaligned16(out))
    return niti_fail(ctx, NITI_ERR_ARG, "niti_linear_fwd: bad argument (pointers must be 16-byte aligned)");
  GemmProblem p;
  fill_fc(p, GK_FC_FWD, M, N, K);
  p.p0 = a; p.p1 = w;
  int64_t dims[3] = {M, N, K};
  char *pad_mem = (char *)ws + NITI_WS_HEADER + round_up((size_t)M * N * 4, 256);
  const size_t need = niti_workspace_bytes(NITI_OP_LINEAR_FWD, dims, 3);
  if (ws && !((uintptr_t)ws & 255) && ws_bytes >= need) {
    const RoundSpec rs = {out, nullptr, 7, round_mode, relu, s_a, s_w, s_out, b_out, nullptr, nullptr};
    const int rc = niti_small_gemm(ctx, (cudaStream_t)stream, ws, p, rs, nullptr, nullptr);
    if (rc != NITI_ERR_SHAPE) return rc;
  }
  return run_gemm_round(ctx, (cudaStream_t)stream, p, ws, ws_bytes, need, pad_mem, out, 7, round_mode, relu,
                        nullptr, s_a, s_w, s_out, b_out);
}

// Backward pass of a fully connected layer; `g` receives the rounded weight gradient, or, with
// update_w, the gradient is subtracted from update_w (= w) in place after the error of the layer
// below has been computed from the old weights.
static int linear_bwd_impl(niti_ctx *ctx, void *stream, const int8_t *a, const int8_t *e, const int8_t *w,
                           int8_t *e_prev, const int8_t *relu_mask_src, int8_t *g, int8_t *update_w,
                           int32_t *b_e, int32_t *b_g, int M, int N, int K, int m_u, int round_mode, void *ws,
                           size_t ws_bytes, const char *who) {
  if (!ctx) return NITI_ERR_ARG;
  if (!a || !e || !w || (!g && !update_w) || M <= 0 || N <= 0 || K <= 0 || m_u < 1 || m_u > 7 ||
      (round_mode != 0 && round_mode != 1) || misaligned16(a) || misaligned16(e) || misaligned16(w) ||
      misaligned16(g) || misaligned16(e_prev) || misaligned16(relu_mask_src)) {
    snprintf(ctx->err, sizeof(ctx->err), "%s: bad argument (pointers must be 16-byte aligned)", who);
    return NITI_ERR_ARG;
  }
  int64_t dims[3] = {M, N, K};
  const size_t need_base = niti_workspace_bytes(NITI_OP_LINEAR_BWD, dims, 3);
  const size_t need = update_w ? niti_workspace_bytes(NITI_OP_LINEAR_BWD_UPDATE, dims, 3) : need_base;
  if (!ws || ((uintptr_t)ws & 255) || ws_bytes < need)
    return niti_fail(ctx, NITI_ERR_WORKSPACE, "workspace missing, misaligned or too small");
  if (update_w) g = (int8_t *)((char *)ws + need_base);       // scratch, used only if the multiply rounds by itself
  // rows padded for TMA: e (shared by both multiplies), then w (error) and a (weight gradient)
  char *pad_mem = (char *)ws + NITI_WS_HEADER + round_up(linear_bwd_acc_elems(M, N, K) * 4, 256);
  GemmProblem pd, pw;
  fill_fc(pd, GK_FC_DGRAD, M, N, K);
  pd.p0 = e; pd.p1 = w;
  fill_fc(pw, GK_FC_WGRAD, M, N, K);
  pw.p0 = e; pw.p1 = a;
  const auto replaces = [&](const int8_t *operand, int width) {
    const uintptr_t out = (uintptr_t)e_prev, in = (uintptr_t)operand;
    return out < in + (uintptr_t)M * (uintptr_t)width && in < out + (uintptr_t)M * (uintptr_t)K;
  };
  const bool in_place = e_prev && (replaces(a, K) || replaces(e, N));      // (an operand of the gradient, too)
  {
    const RoundSpec rd = {e_prev, relu_mask_src, 7, round_mode, 0, nullptr, nullptr, nullptr, b_e, nullptr, nullptr};
    const RoundSpec rw = {g, nullptr, m_u, round_mode, 0, nullptr, nullptr, nullptr, b_g, nullptr, update_w};
    // One launch runs both multiplies at once: an error that replaces the layer's input or the error above it is left to the
    // launches below, which read them for the weight gradient before they write the error.
    int rc = NITI_ERR_SHAPE;
    if (!e_prev) rc = niti_small_gemm(ctx, (cudaStream_t)stream, ws, pw, rw, nullptr, nullptr);
    else if (!in_place) rc = niti_small_gemm(ctx, (cudaStream_t)stream, ws, pd, rd, &pw, &rw);
    if (rc != NITI_ERR_SHAPE) return rc;
  }
  char *pad_a = pad_mem + pad_bytes(pd) - pad_bytes(pw, 0);      // (the weight gradient finds e padded already)
  if (pad_bytes(pd, 0) && N >= 32 && ctx->engine != 1) {
    const int rcp = niti_launch_pad_pitch(ctx, (cudaStream_t)stream, e, (int8_t *)pad_mem, M, N, pitch16(N));
    if (rcp != NITI_OK) return rcp;
    pd.q0 = pw.q0 = (int8_t *)pad_mem;
    pd.ld0 = pw.ld0 = pitch16(N);
  }
  const auto error_below = [&]() {
    return run_gemm_round(ctx, (cudaStream_t)stream, pd, ws, ws_bytes, need, pad_mem, e_prev, 7, round_mode, 0, relu_mask_src,
                          nullptr, nullptr, nullptr, b_e);
  };
  // The error below needs the weights as they were, the gradient its operands as they were: beside an error that replaces one
  // of them the gradient is kept until the error is there.
  const bool error_first = e_prev && update_w && !in_place;
  int rc = error_first ? error_below() : NITI_OK;
  if (rc == NITI_OK)
    rc = run_gemm_round(ctx, (cudaStream_t)stream, pw, ws, ws_bytes, need, pad_a, g, m_u, round_mode, 0, nullptr, nullptr, nullptr,
                        nullptr, b_g, in_place ? nullptr : update_w);
  if (rc != NITI_OK || !e_prev || error_first) return rc;
  rc = error_below();
  return rc == NITI_OK && update_w ? niti_launch_sgd_update(ctx, (cudaStream_t)stream, update_w, g, (long long)N * K) : rc;
}

extern "C" int niti_linear_bwd(niti_ctx *ctx, void *stream, const int8_t *a, const int8_t *e,
                               const int8_t *w, int8_t *e_prev, const int8_t *relu_mask_src, int8_t *g,
                               int32_t *b_e, int32_t *b_g, int M, int N, int K, int m_u, int round_mode,
                               void *ws, size_t ws_bytes) {
  if (ctx && !g) return niti_fail(ctx, NITI_ERR_ARG, "niti_linear_bwd: bad argument (g is null)");
  return linear_bwd_impl(ctx, stream, a, e, w, e_prev, relu_mask_src, g, nullptr, b_e, b_g, M, N, K, m_u,
                         round_mode, ws, ws_bytes, "niti_linear_bwd");
}

extern "C" int niti_linear_bwd_update(niti_ctx *ctx, void *stream, const int8_t *a, const int8_t *e, int8_t *w,
                                      int8_t *e_prev, const int8_t *relu_mask_src, int32_t *b_e, int32_t *b_g,
                                      int M, int N, int K, int m_u, int round_mode, void *ws, size_t ws_bytes) {
  return linear_bwd_impl(ctx, stream, a, e, w, e_prev, relu_mask_src, nullptr, w, b_e, b_g, M, N, K, m_u,
                         round_mode, ws, ws_bytes, "niti_linear_bwd_update");
}

// padded operands of a convolution call that gathers nothing: right behind the accumulators
static inline char *conv_pad_mem(const GemmProblem &p, void *ws) {
  return (char *)ws + NITI_WS_HEADER + round_up((size_t)(p.gm * p.gn) * 4, 256);
}

static int conv_args_ok(int B, int H, int W, int Ci, int Co, int R, int S, int pad, int round_mode) {
  return B > 0 && H > 0 && W > 0 && Ci > 0 && Co > 0 && R > 0 && S > 0 && pad >= 0 &&
         (round_mode == 0 || round_mode == 1);
}

static int conv_fwd_impl(niti_ctx *ctx, void *stream, const int8_t *x, const int32_t *s_x, const int8_t *w,
                         const int32_t *s_w, int8_t *y, int8_t *y_pool, int32_t *s_y, int32_t *b_y, int B, int H,
                         int W, int Cin, int Cout, int R, int S, int pad, int stride, int relu, int round_mode,
                         void *ws, size_t ws_bytes) {
  if (!ctx) return NITI_ERR_ARG;
  GemmProblem p;
  memset(&p, 0, sizeof(p));
  if (!x || !w || !y || !s_x || !s_w || !conv_args_ok(B, H, W, Cin, Cout, R, S, pad, round_mode) ||
      misaligned16(x) || misaligned16(w) || misaligned16(y) ||
      !fill_conv(p, GK_CONV_FWD, B, H, W, Cin, Cout, R, S, pad, stride))
    return niti_fail(ctx, NITI_ERR_ARG, "niti_conv_fwd: bad argument (pointers must be 16-byte aligned)");
  p.p0 = x; p.p1 = w;
  int64_t dims[9] = {B, H, W, Cin, Cout, R, S, pad, stride};
  const size_t need = niti_workspace_bytes(NITI_OP_CONV_FWD, dims, 9);
  const WindowGeometry wg = window_geometry(p);
  if (wg.Cp && ctx->engine != 1 && ws && !((uintptr_t)ws & 255) && ws_bytes >= need) {
    int8_t *xw = (int8_t *)conv_pad_mem(p, ws), *ww = xw + wg.x_bytes;
    const int rc = niti_launch_widen(ctx, (cudaStream_t)stream, x, xw, B * H, W, Cin, wg.Cp, pad, wg.row_bytes, w, ww, Cout * R, S,
                                     wg.pitch);
    if (rc != NITI_OK) return rc;
    GemmProblem q = window_problem(p, wg, xw);
    q.q1 = ww;
    return run_gemm_round(ctx, (cudaStream_t)stream, p, ws, ws_bytes, need, nullptr, y, 7, round_mode, relu, nullptr, s_x, s_w,
                          s_y, b_y, nullptr, y_pool, &q);
  }
  if (few_channel_conv(Cin, R, S) && ctx->engine != 1) {
    if (!ws || ((uintptr_t)ws & 255) || ws_bytes < need)
      return niti_fail(ctx, NITI_ERR_WORKSPACE, "workspace missing, misaligned or too small");
    // gather the taps into [M][32] rows, pad the weights to [Cout][32], then a K = 32 multiply
    cudaStream_t st = (cudaStream_t)stream;
    const size_t M = (size_t)p.gm;
    char *base = (char *)ws + NITI_WS_HEADER + round_up(M * (size_t)Cout * 4, 256);
    int8_t *xcol = (int8_t *)base;
    int8_t *wcol = (int8_t *)(base + round_up(M * 32, 256));
    if (ctx->tap_buf && M * 32 <= ctx->tap_bytes) {
      // gathered into the caller's tap cache: the weight-gradient call of this layer finds the rows there
      xcol = ctx->tap_buf;
      ctx->tap_x = x;
      const int dims[9] = {B, H, W, Cin, R, S, pad, stride, 1};
      memcpy(ctx->tap_dims, dims, sizeof(dims));
    }
    int rc = niti_launch_im2col32(ctx, st, x, xcol, B, H, W, Cin, R, S, pad, stride, p.Ho, p.Wo);
    if (rc == NITI_OK) rc = niti_launch_pad_pitch(ctx, st, w, wcol, Cout, R * S * Cin, 32);
    if (rc != NITI_OK) return rc;
    GemmProblem q;
    fill_fc(q, GK_FC_FWD, (int)M, Cout, 32);
    q.p0 = xcol; q.p1 = wcol;
    rc = run_gemm_round(ctx, st, q, ws, ws_bytes, need, nullptr, y, 7, round_mode, relu, nullptr, s_x, s_w, s_y, b_y);
    if (rc != NITI_OK || !y_pool) return rc;
    return niti_launch_maxpool2_fwd(ctx, st, y, y_pool, B, p.Ho, p.Wo, Cout);
  }
  return run_gemm_round(ctx, (cudaStream_t)stream, p, ws, ws_bytes, need, conv_pad_mem(p, ws), y, 7, round_mode, relu, nullptr,
                        s_x, s_w, s_y, b_y, nullptr, y_pool);
}

extern "C" int niti_conv_fwd_strided(niti_ctx *ctx, void *stream, const int8_t *x, const int32_t *s_x,
                                     const int8_t *w, const int32_t *s_w, int8_t *y, int32_t *s_y, int32_t *b_y,
                                     int B, int H, int W, int Cin, int Cout, int R, int S, int pad, int stride,
                                     int relu, int round_mode, void *ws, size_t ws_bytes) {
  return conv_fwd_impl(ctx, stream, x, s_x, w, s_w, y, nullptr, s_y, b_y, B, H, W, Cin, Cout, R, S, pad, stride, relu,
                       round_mode, ws, ws_bytes);
}

extern "C" int niti_conv_fwd_pool(niti_ctx *ctx, void *stream, const int8_t *x, const int32_t *s_x, const int8_t *w,
                                  const int32_t *s_w, int8_t *y, int8_t *y_pool, int32_t *s_y, int32_t *b_y, int B,
                                  int H, int W, int Cin, int Cout, int R, int S, int pad, int relu, int round_mode,
                                  void *ws, size_t ws_bytes) {
  if (!ctx) return NITI_ERR_ARG;
  const int Ho = H + 2 * pad - R + 1, Wo = W + 2 * pad - S + 1;
  if (!y_pool || Ho <= 0 || Wo <= 0 || (Ho & 1) || (Wo & 1) || misaligned16(y_pool))
    return niti_fail(ctx, NITI_ERR_ARG, "niti_conv_fwd_pool: bad argument (output height and width must be even)");
  return conv_fwd_impl(ctx, stream, x, s_x, w, s_w, y, y_pool, s_y, b_y, B, H, W, Cin, Cout, R, S, pad, 1, relu,
                       round_mode, ws, ws_bytes);
}

extern "C" int niti_conv_fwd(niti_ctx *ctx, void *stream, const int8_t *x, const int32_t *s_x,
                             const int8_t *w, const int32_t *s_w, int8_t *y, int32_t *s_y, int32_t *b_y,
                             int B, int H, int W, int Cin, int Cout, int R, int S, int pad, int relu,
                             int round_mode, void *ws, size_t ws_bytes) {
  return niti_conv_fwd_strided(ctx, stream, x, s_x, w, s_w, y, s_y, b_y, B, H, W, Cin, Cout, R, S, pad, 1, relu,
                               round_mode, ws, ws_bytes);
}

extern "C" int niti_conv_dgrad_strided(niti_ctx *ctx, void *stream, const int8_t *e, const int8_t *w,
                                       int8_t *e_prev, const int8_t *relu_mask_src, int32_t *b_e, int B, int H,
                                       int W, int Cin, int Cout, int R, int S, int pad, int stride, int round_mode,
                                       void *ws, size_t ws_bytes) {
  if (!ctx) return NITI_ERR_ARG;
  GemmProblem p;
  memset(&p, 0, sizeof(p));
  if (!e || !w || !e_prev || !conv_args_ok(B, H, W, Cin, Cout, R, S, pad, round_mode) || misaligned16(e) ||
      misaligned16(w) || misaligned16(e_prev) || misaligned16(relu_mask_src) ||
      !fill_conv(p, GK_CONV_DGRAD, B, H, W, Cin, Cout, R, S, pad, stride))
    return niti_fail(ctx, NITI_ERR_ARG, "niti_conv_dgrad: bad argument (pointers must be 16-byte aligned)");
  p.p0 = e; p.p1 = w;
  int64_t dims[9] = {B, H, W, Cin, Cout, R, S, pad, stride};
  return run_gemm_round(ctx, (cudaStream_t)stream, p, ws, ws_bytes,
                        niti_workspace_bytes(NITI_OP_CONV_DGRAD, dims, 9), conv_pad_mem(p, ws), e_prev, 7, round_mode, 0,
                        relu_mask_src, nullptr, nullptr, nullptr, b_e);
}

extern "C" int niti_conv_dgrad(niti_ctx *ctx, void *stream, const int8_t *e, const int8_t *w,
                               int8_t *e_prev, const int8_t *relu_mask_src, int32_t *b_e, int B, int H,
                               int W, int Cin, int Cout, int R, int S, int pad, int round_mode, void *ws,
                               size_t ws_bytes) {
  return niti_conv_dgrad_strided(ctx, stream, e, w, e_prev, relu_mask_src, b_e, B, H, W, Cin, Cout, R, S, pad, 1,
                                 round_mode, ws, ws_bytes);
}

// Weight gradient of a convolution; with update_w the rounded gradient is subtracted from the
// weights in place instead of being returned.
static int conv_wgrad_impl(niti_ctx *ctx, void *stream, const int8_t *x, const int8_t *e, int8_t *g,
                           int8_t *update_w, int32_t *b_g, int B, int H, int W, int Cin, int Cout, int R, int S,
                           int pad, int stride, int m_u, int round_mode, void *ws, size_t ws_bytes, const char *who) {
  if (!ctx) return NITI_ERR_ARG;
  GemmProblem p;
  memset(&p, 0, sizeof(p));
  if (!x || !e || (!g && !update_w) || m_u < 1 || m_u > 7 || !conv_args_ok(B, H, W, Cin, Cout, R, S, pad, round_mode) ||
      misaligned16(x) || misaligned16(e) || misaligned16(g) || misaligned16(update_w) ||
      !fill_conv(p, GK_CONV_WGRAD, B, H, W, Cin, Cout, R, S, pad, stride)) {
    snprintf(ctx->err, sizeof(ctx->err), "%s: bad argument (pointers must be 16-byte aligned)", who);
    return NITI_ERR_ARG;
  }
  p.p0 = e; p.p1 = x;
  int64_t dims[9] = {B, H, W, Cin, Cout, R, S, pad, stride};
  const size_t need_base = niti_workspace_bytes(NITI_OP_CONV_WGRAD, dims, 9);
  const size_t need = update_w ? niti_workspace_bytes(NITI_OP_CONV_WGRAD_UPDATE, dims, 9) : need_base;
  if (!ws || ((uintptr_t)ws & 255) || ws_bytes < need)
    return niti_fail(ctx, NITI_ERR_WORKSPACE, "workspace missing, misaligned or too small");
  if (update_w) g = (int8_t *)((char *)ws + need_base);       // scratch, used only where the rounding stores int8
  const WindowGeometry wg = window_geometry(p);
  const bool own_form = (wg.Cp || few_channel_conv(Cin, R, S)) && ctx->engine != 1;
  if (own_form) {
    // the multiply leaves int32 sums over widened windows (columns r, s * Cp + c) or over gathered 32-byte rows; the
    // columns that are taps are then rounded into g, or subtracted from the weights
    cudaStream_t st = (cudaStream_t)stream;
    const size_t M = (size_t)B * p.Ho * p.Wo;
    WsHeader *hdr = niti_take_header(ctx, st, ws);
    int rc = NITI_OK;
    int8_t *xcol = (int8_t *)conv_pad_mem(p, ws);
    const size_t x_bytes = wg.Cp ? wg.x_bytes + wg.w_bytes : round_up(M * 32, 256) + round_up((size_t)Cout * 32, 256);
    int32_t *acc = (int32_t *)(xcol + x_bytes);
    const int acc_pitch = wg.Cp ? R * wg.pitch : 32;
    char *pad_mem = (char *)acc + round_up((size_t)Cout * acc_pitch * 4, 256);
    GemmProblem q;
    if (wg.Cp) {
      rc = niti_launch_widen(ctx, st, x, xcol, B * H, W, Cin, wg.Cp, pad, wg.row_bytes, nullptr, nullptr, 0, S, wg.pitch);
      q = window_problem(p, wg, xcol);
    } else {
      if (tap_cache_hit(ctx, x, B, H, W, Cin, R, S, pad, stride)) {
        xcol = ctx->tap_buf;               // gathered by the forward call
        ctx->tap_dims[8] = 0;              // (used once: the next forward call fills the cache again)
      } else rc = niti_launch_im2col32(ctx, st, x, xcol, B, H, W, Cin, R, S, pad, stride, p.Ho, p.Wo);
      fill_fc(q, GK_FC_WGRAD, (int)M, Cout, 32);     // rows M are the contraction
      q.p0 = e; q.p1 = xcol;
    }
    if (rc != NITI_OK) return rc;
    rc = pad_operands(ctx, st, q, pad_mem, (const char *)ws + need_base);
    if (rc != NITI_OK) return rc;
    bool fused = false;
    RoundSpec none = {nullptr, nullptr, m_u, round_mode, 0, nullptr, nullptr, nullptr, nullptr, nullptr};
    rc = niti_tc_gemm(ctx, st, q, none, acc, hdr, &fused);       // (no output: int32 accumulators)
    if (rc == NITI_ERR_SHAPE && !wg.Cp) {
      rc = niti_simt_gemm(ctx, st, q, acc, hdr);
      if (rc == NITI_OK) rc = niti_reduce_after_gemm(ctx, st, q.kind, acc, (long long)Cout * 32, hdr);
    }
    if (rc == NITI_OK)
      return niti_launch_round_compact(ctx, st, acc, hdr, g, Cout, R * S * Cin, acc_pitch, S * Cin, wg.Cp ? wg.pitch : S * Cin,
                                       Cin, wg.Cp ? wg.Cp : Cin, m_u, round_mode, b_g, update_w);
    if (rc != NITI_ERR_SHAPE) return rc;
  }
  return run_gemm_round(ctx, (cudaStream_t)stream, p, ws, ws_bytes, need, conv_pad_mem(p, ws), g, m_u, round_mode, 0, nullptr,
                        nullptr, nullptr, nullptr, b_g, update_w, nullptr, nullptr, own_form);
}

extern "C" int niti_conv_wgrad_strided(niti_ctx *ctx, void *stream, const int8_t *x, const int8_t *e, int8_t *g,
                                       int32_t *b_g, int B, int H, int W, int Cin, int Cout, int R, int S, int pad,
                                       int stride, int m_u, int round_mode, void *ws, size_t ws_bytes) {
  if (ctx && !g) return niti_fail(ctx, NITI_ERR_ARG, "niti_conv_wgrad: bad argument (g is null)");
  return conv_wgrad_impl(ctx, stream, x, e, g, nullptr, b_g, B, H, W, Cin, Cout, R, S, pad, stride, m_u, round_mode,
                         ws, ws_bytes, "niti_conv_wgrad");
}

extern "C" int niti_conv_wgrad(niti_ctx *ctx, void *stream, const int8_t *x, const int8_t *e, int8_t *g,
                               int32_t *b_g, int B, int H, int W, int Cin, int Cout, int R, int S, int pad,
                               int m_u, int round_mode, void *ws, size_t ws_bytes) {
  return niti_conv_wgrad_strided(ctx, stream, x, e, g, b_g, B, H, W, Cin, Cout, R, S, pad, 1, m_u, round_mode, ws,
                                 ws_bytes);
}

extern "C" int niti_conv_wgrad_update(niti_ctx *ctx, void *stream, const int8_t *x, const int8_t *e, int8_t *w,
                                      int32_t *b_g, int B, int H, int W, int Cin, int Cout, int R, int S, int pad,
                                      int m_u, int round_mode, void *ws, size_t ws_bytes) {
  if (ctx && !w) return niti_fail(ctx, NITI_ERR_ARG, "niti_conv_wgrad_update: bad argument (w is null)");
  return conv_wgrad_impl(ctx, stream, x, e, nullptr, w, b_g, B, H, W, Cin, Cout, R, S, pad, 1, m_u, round_mode, ws,
                         ws_bytes, "niti_conv_wgrad_update");
}
