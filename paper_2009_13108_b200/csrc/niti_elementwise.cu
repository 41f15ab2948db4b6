// HBM-bound kernels of the NITI library: the shift-and-round pass (Algorithm 2/3), the integer
// cross-entropy gradient (Section 3.5), the weight update (Algorithm 1) and the int8 support ops.
#include "niti_common.cuh"
#include <mutex>

// ---------------------------------------------------------------------------------------------
// Shift-and-round pass over an int32 accumulator tensor (Algorithm 2, with Algorithm 3 rounding).
// Every thread handles 16 consecutive elements: four 16-byte loads, one 16-byte store.
// ---------------------------------------------------------------------------------------------
__device__ __forceinline__ unsigned sat_sub_clamp127(unsigned w, unsigned g) {
  // per byte: clamp(w - g, -127, 127): saturating subtract gives [-128, 127]; lift -128 to -127
  return __vmaxs4(__vsubss4(w, g), 0x81818181u);
}

__global__ void __launch_bounds__(256)
round_i32_kernel(const int32_t *__restrict__ acc, const WsHeader *__restrict__ hdr,
                 int8_t *__restrict__ out, long long n, int mbits, int round_mode, int relu,
                 const int8_t *__restrict__ mask, const int32_t *__restrict__ s_a,
                 const int32_t *__restrict__ s_w, int32_t *__restrict__ s_out,
                 int32_t *__restrict__ b_out, uint32_t *__restrict__ status, int8_t *__restrict__ upd_w) {
  niti_enter(acc, hdr, mask, s_a, s_w, upd_w);
  const int b = niti_bitlen32(hdr->maxabs32);
  const int bp = b > mbits ? b - mbits : 0;
  const unsigned qmax = (1u << mbits) - 1u;
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    if (b_out) *b_out = b;
    if (s_out) {
      int s = bp + (s_a ? *s_a : 0) + (s_w ? *s_w : 0);
      *s_out = s;
      if (s < -128 || s > 127) atomicOr(status, NITI_DEV_EXP_RANGE);
    }
  }
  const long long nvec = n >> 4;
  const long long stride = (long long)gridDim.x * blockDim.x;
  for (long long v = (long long)blockIdx.x * blockDim.x + threadIdx.x; v < nvec; v += stride) {
    const int4 *src = reinterpret_cast<const int4 *>(acc) + v * 4;
    int4 x0 = __ldcs(src), x1 = __ldcs(src + 1), x2 = __ldcs(src + 2), x3 = __ldcs(src + 3);
    int xs[16] = {x0.x, x0.y, x0.z, x0.w, x1.x, x1.y, x1.z, x1.w,
                  x2.x, x2.y, x2.z, x2.w, x3.x, x3.y, x3.z, x3.w};
    int4 mk = make_int4(-1, -1, -1, -1);
    if (mask) {
      int4 mv = *(reinterpret_cast<const int4 *>(mask) + v);
      mk.x = __vcmpgts4(mv.x, 0); mk.y = __vcmpgts4(mv.y, 0);
      mk.z = __vcmpgts4(mv.z, 0); mk.w = __vcmpgts4(mv.w, 0);
    }
    unsigned o[4];
#pragma unroll
    for (int w = 0; w < 4; ++w) {
      unsigned word = 0;
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        int q = niti_round_i32(xs[w * 4 + j], bp, qmax, round_mode);
        if (relu && q < 0) q = 0;
        word |= (unsigned)(q & 0xff) << (8 * j);
      }
      o[w] = word;
    }
    int4 ov = make_int4(o[0] & mk.x, o[1] & mk.y, o[2] & mk.z, o[3] & mk.w);
    if (upd_w) {
      // weight update fused with the rounding of the weight gradient (Section 3.3: the rounded
      // gradient is never stored): w <- clamp(w - q, -127, 127)
      int4 wv = *(reinterpret_cast<int4 *>(upd_w) + v);
      wv.x = sat_sub_clamp127(wv.x, ov.x); wv.y = sat_sub_clamp127(wv.y, ov.y);
      wv.z = sat_sub_clamp127(wv.z, ov.z); wv.w = sat_sub_clamp127(wv.w, ov.w);
      *(reinterpret_cast<int4 *>(upd_w) + v) = wv;
    } else {
      *(reinterpret_cast<int4 *>(out) + v) = ov;
    }
  }
  // ragged tail (fewer than 16 elements)
  long long t = (nvec << 4) + (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (t < n) {
    int q = niti_round_i32(acc[t], bp, qmax, round_mode);
    if (relu && q < 0) q = 0;
    if (mask && mask[t] <= 0) q = 0;
    if (upd_w) {
      int d = (int)upd_w[t] - q;
      upd_w[t] = (int8_t)(d > 127 ? 127 : (d < -127 ? -127 : d));
    } else {
      out[t] = (int8_t)q;
    }
  }
}

int niti_launch_round(niti_ctx *ctx, cudaStream_t st, const int32_t *acc, const WsHeader *hdr,
                      int8_t *out, long long n, int mbits, int round_mode, int relu,
                      const int8_t *mask, const int32_t *s_a, const int32_t *s_w, int32_t *s_out,
                      int32_t *b_out, int8_t *upd_w) {
  long long nvec = n >> 4;
  long long blocks = (nvec + 255) / 256;
  long long cap = (long long)ctx->sm_count * 16;
  if (blocks > cap) blocks = cap;
  if (blocks < 1) blocks = 1;
  niti_launch(st, (unsigned)blocks, 256, 0, round_i32_kernel, acc, hdr, out, n, mbits, round_mode, relu, mask,
                                                     s_a, s_w, s_out, b_out, ctx->d_status, upd_w);
  ctx->launches++;
  NITI_CUDA_TRY(ctx, cudaGetLastError());
  return NITI_OK;
}

// ---------------------------------------------------------------------------------------------
// Few-channel convolutions (first layer: 1 or 3 input channels, R*S*Cin <= 32): the taps of every
// output pixel are gathered into one 32-byte row so that the layer becomes a plain K = 32 matrix
// multiply for the tensor-core engine.  Column k = (r * S + s) * Cin + ci, zero beyond R*S*Cin.
// ---------------------------------------------------------------------------------------------
__global__ void __launch_bounds__(256)
im2col32_kernel(const int8_t *__restrict__ x, int8_t *__restrict__ xcol, int B, int H, int W, int Ci, int R,
                int S, int pad, int stride, int Ho, int Wo) {
  niti_enter(x);
  const long long M = (long long)B * Ho * Wo;
  for (long long m = (long long)blockIdx.x * blockDim.x + threadIdx.x; m < M;
       m += (long long)gridDim.x * blockDim.x) {
    const int j = (int)(m % Wo);
    const long long t = m / Wo;
    const int i = (int)(t % Ho);
    const long long b = t / Ho;
    unsigned w[8] = {0, 0, 0, 0, 0, 0, 0, 0};
    int k = 0;
    for (int r = 0; r < R; ++r) {
      const int ii = i * stride + r - pad;
      for (int q = 0; q < S; ++q) {
        const int jj = j * stride + q - pad;
        const bool in = ii >= 0 && ii < H && jj >= 0 && jj < W;
        const int8_t *src = x + ((b * H + ii) * W + jj) * Ci;
        for (int c = 0; c < Ci; ++c, ++k) {
          const unsigned v = in ? (unsigned)(uint8_t)src[c] : 0u;
          w[k >> 2] |= v << (8 * (k & 3));
        }
      }
    }
    int4 *dst = reinterpret_cast<int4 *>(xcol + m * 32);
    dst[0] = make_int4(w[0], w[1], w[2], w[3]);
    dst[1] = make_int4(w[4], w[5], w[6], w[7]);
  }
}

// Fast path for the RGB first layer (Cin = 3, 3x3 taps, pad 1, W % 4 == 0): one block per output image
// row stages the three input rows in shared memory (one pixel of zero halo on each side) and every
// thread assembles the 27-byte tap vectors of four consecutive pixels from five aligned words per
// row, with byte offsets known at compile time.  The generic kernel above issues 27 byte loads per
// pixel and ran at a fifth of the memory rate.
__device__ __forceinline__ unsigned win_byte(const unsigned (&w)[5], int idx) {
  return (w[idx >> 2] >> (8 * (idx & 3))) & 0xffu;
}
__global__ void __launch_bounds__(128)
im2col32_rgb3x3_kernel(const int8_t *__restrict__ x, int8_t *__restrict__ xcol, int B, int H, int W) {
  niti_enter(x);
  extern __shared__ unsigned rgb_rows[];          // 3 rows x pitch words
  const int row_words = W * 3 / 4;                // data words per image row
  const int pitch = row_words + 2;                // one halo word on each side (3 of its 4 bytes are used)
  const int i = blockIdx.x % H;
  const long long b = blockIdx.x / H;
  for (int idx = threadIdx.x; idx < 3 * pitch; idx += blockDim.x) {
    const int r = idx / pitch, c = idx % pitch - 1;
    const int ii = i + r - 1;
    unsigned v = 0;
    if (c >= 0 && c < row_words && ii >= 0 && ii < H)
      v = reinterpret_cast<const unsigned *>(x + (b * H + ii) * (long long)W * 3)[c];
    rgb_rows[idx] = v;
  }
  __syncthreads();
  // pixel j of a staged row starts at byte 4 + 3 j; the window of pixels 4t-1 .. 4t+4 starts at
  // byte 12 t + 1, i.e. at byte 1 of word 3 t
  for (int t = threadIdx.x; t < W / 4; t += blockDim.x) {
    unsigned win[3][5];
#pragma unroll
    for (int r = 0; r < 3; ++r)
#pragma unroll
      for (int k = 0; k < 5; ++k) win[r][k] = rgb_rows[r * pitch + 3 * t + k];
    int4 *dst = reinterpret_cast<int4 *>(xcol + ((b * H + i) * (long long)W + 4 * t) * 32);
#pragma unroll
    for (int px = 0; px < 4; ++px) {
      unsigned o[8];
#pragma unroll
      for (int wd = 0; wd < 8; ++wd) {
        unsigned v = 0;
#pragma unroll
        for (int by = 0; by < 4; ++by) {
          const int k = 4 * wd + by;              // column of the gathered row: (tap row, tap col, channel)
          if (k < 27) v |= win_byte(win[k / 9], 1 + 3 * px + k % 9) << (8 * by);
        }
        o[wd] = v;
      }
      // one gathered row = one 32-byte sector: a single 256-bit store per pixel
      asm volatile("st.global.v8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};"
                   ::"l"(dst + 2 * px), "r"(o[0]), "r"(o[1]), "r"(o[2]), "r"(o[3]), "r"(o[4]), "r"(o[5]), "r"(o[6]), "r"(o[7])
                   : "memory");
    }
  }
}

__global__ void __launch_bounds__(256)
clear_kernel(int8_t *p, unsigned vecs, unsigned bytes) {
  niti_enter(p);
  for (unsigned i = blockIdx.x * blockDim.x + threadIdx.x; i < vecs; i += gridDim.x * blockDim.x)
    reinterpret_cast<int4 *>(p)[i] = make_int4(0, 0, 0, 0);
  const unsigned tail = vecs * 16u + 4u * threadIdx.x;
  if (blockIdx.x == 0 && tail < bytes) *reinterpret_cast<int *>(p + tail) = 0;
}

int niti_memset0(niti_ctx *ctx, cudaStream_t st, void *p, size_t bytes) {
  ctx->launches++;
  if (bytes >= ((size_t)1 << 31) || (bytes & 3) || ((uintptr_t)p & 15)) {
    NITI_CUDA_TRY(ctx, cudaMemsetAsync(p, 0, bytes, st));
    return NITI_OK;
  }
  const unsigned vecs = (unsigned)(bytes >> 4);
  unsigned blocks = (vecs + 255u) / 256u;
  const unsigned most = 8u * (unsigned)ctx->sm_count;
  blocks = blocks < 1u ? 1u : (blocks > most ? most : blocks);
  NITI_CUDA_TRY(ctx, niti_launch(st, blocks, 256, 0, clear_kernel, (int8_t *)p, vecs, (unsigned)bytes));
  return NITI_OK;
}

// Rows of n bytes -> rows of `pitch` bytes (a multiple of 16, pitch >= n), zero padded.  Sixteen output bytes per thread
// from the aligned source words around them (bound: latency; for 4096 rows of 1000 bytes one byte per thread took 12.9 us,
// one output word 6.6 us, this 3.3 us less in the call it belongs to).  src and dst are 16-byte aligned.
__global__ void __launch_bounds__(256)
pad_pitch_kernel(const int8_t *__restrict__ src, int8_t *__restrict__ dst, long long rows, int n, int pitch) {
  niti_enter(src);
  const unsigned parts = (unsigned)pitch >> 4;
  for (long long base = (long long)blockIdx.x * blockDim.x; base < rows * parts; base += (long long)gridDim.x * blockDim.x) {
    // (the division is by thread and 32 bits wide: the block's first row is found once)
    const long long r0 = base / parts;
    const unsigned t = (unsigned)(base - r0 * parts) + threadIdx.x, dr = t / parts, part = t - dr * parts;
    const long long r = r0 + dr;
    if (r >= rows) continue;
    const int left = n - 16 * (int)part;                  // valid bytes of this part
    const long long o = r * n + 16 * part;
    const int mis = (int)(o & 3);
    const unsigned *p = reinterpret_cast<const unsigned *>(src) + (o >> 2);
    unsigned v[5], out[4];
#pragma unroll
    for (int k = 0; k < 5; ++k) v[k] = left > 0 && 4 * k < mis + (left < 16 ? left : 16) ? p[k] : 0u;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const int have = left - 4 * k;
      const unsigned w = __funnelshift_r(v[k], v[k + 1], 8u * (unsigned)mis);
      out[k] = have >= 4 ? w : (have <= 0 ? 0u : w & (0xffffffffu >> (32 - 8 * have)));
    }
    *reinterpret_cast<uint4 *>(dst + r * pitch + 16 * part) = make_uint4(out[0], out[1], out[2], out[3]);
  }
}

int niti_launch_pad_pitch(niti_ctx *ctx, cudaStream_t st, const int8_t *src, int8_t *dst, long long rows, int n, int pitch) {
  long long blocks = (rows * (pitch >> 4) + 255) / 256;
  if (blocks > (long long)ctx->sm_count * 16) blocks = (long long)ctx->sm_count * 16;
  niti_launch(st, (unsigned)blocks, 256, 0, pad_pitch_kernel, src, dst, rows, n, pitch);
  ctx->launches++;
  NITI_CUDA_TRY(ctx, cudaGetLastError());
  return NITI_OK;
}

// Rounds the columns of acc[rows][pitch] (int32) that hold taps: out[rows][taps * rowk], or subtracts them from
// upd_w.  Column of tap row r, column s, channel c: r * rpitch + s * Cp + c.
__global__ void __launch_bounds__(256)
round_compact_kernel(const int32_t *__restrict__ acc, const WsHeader *__restrict__ hdr, int8_t *__restrict__ out,
                     int rows, int k, int pitch, int rowk, int rpitch, int Ci, int Cp, int mbits, int round_mode,
                     int32_t *__restrict__ b_out, int8_t *__restrict__ upd_w) {
  niti_enter(acc, hdr, upd_w);
  const int b = niti_bitlen32(hdr->maxabs32);
  const int bp = b > mbits ? b - mbits : 0;
  const unsigned qmax = (1u << mbits) - 1u;
  const int idx = blockIdx.x * blockDim.x + threadIdx.x;
  if (idx == 0 && b_out) *b_out = b;
  if (idx < rows * k) {
    const int row = idx / k, c = idx - row * k;
    const int r = c / rowk, rem = c - r * rowk, sx = rem / Ci, ci = rem - sx * Ci;
    const int q = niti_round_i32(acc[(long long)row * pitch + r * rpitch + sx * Cp + ci], bp, qmax, round_mode);
    if (upd_w) {
      const int d = (int)upd_w[idx] - q;
      upd_w[idx] = (int8_t)(d > 127 ? 127 : (d < -127 ? -127 : d));
    } else {
      out[idx] = (int8_t)q;
    }
  }
}

// Few-channel convolutions with more than 32 taps ("windows", see window_geometry): image rows with `pad` zero
// pixels on the left, enough on the right for the last window, and every pixel widened from Ci to Cp bytes (4, 8 or
// 16).  Bound: memory (the taps are not copied, so 224 x 224 x 3 images become 13 MB for an 11 x 11 stride-4 layer where
// gathered rows were 74 MB and took 80 us to write).  A thread writes 16 bytes, 16 / Cp pixels, from unaligned words
// (with a byte per load and a 64-bit division per word the pass took 20 us).
__global__ void __launch_bounds__(256)
widen_pixels_kernel(const int8_t *__restrict__ x, int8_t *__restrict__ xw, unsigned rows, int W, int Ci, int cp_shift, int pad,
                    unsigned row_parts) {
  niti_enter(x);
  const unsigned total = rows * row_parts, stride = gridDim.x * blockDim.x;
  for (unsigned idx = blockIdx.x * blockDim.x + threadIdx.x; idx < total; idx += stride) {
    const unsigned r = idx / row_parts, part = idx - r * row_parts;
    const int8_t *row = x + (long long)r * W * Ci;
    unsigned v[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int byte = (int)part * 16 + 4 * j, px = (byte >> cp_shift) - pad, c0 = byte & ((1 << cp_shift) - 1);
      v[j] = px >= 0 && px < W ? niti_load_bytes4(row + px * Ci + c0, Ci - c0) : 0u;
    }
    reinterpret_cast<uint4 *>(xw)[idx] = make_uint4(v[0], v[1], v[2], v[3]);
  }
}
// weights [Cout][R][S][Ci] -> [Cout][R][pitch], tap column s in bytes s * Cp .. s * Cp + Ci - 1, zero elsewhere
__global__ void __launch_bounds__(256)
widen_weights_kernel(const int8_t *__restrict__ w, int8_t *__restrict__ ww, int rows, int S, int Ci, int Cp, int pitch) {
  niti_enter(w);
  const long long idx = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (idx < (long long)rows * pitch) {
    const int r = (int)(idx / pitch), b = (int)(idx - (long long)r * pitch);
    const int sx = b / Cp, c = b - sx * Cp;
    ww[idx] = (sx < S && c < Ci) ? w[((long long)r * S + sx) * Ci + c] : (int8_t)0;
  }
}
int niti_launch_widen(niti_ctx *ctx, cudaStream_t st, const int8_t *x, int8_t *xw, int rows, int W, int Ci, int Cp, int pad,
                      int row_bytes, const int8_t *w, int8_t *ww, int wrows, int S, int pitch) {
  const long long parts = (long long)rows * (row_bytes / 16);
  if (parts >= (1LL << 31)) return niti_fail(ctx, NITI_ERR_SHAPE, "few-channel convolution: image too large");
  long long blocks = (parts + 255) / 256;
  if (blocks > (long long)ctx->sm_count * 64) blocks = (long long)ctx->sm_count * 64;
  const int cp_shift = Cp == 4 ? 2 : (Cp == 8 ? 3 : 4);
  niti_launch(st, (unsigned)blocks, 256, 0, widen_pixels_kernel, x, xw, (unsigned)rows, W, Ci, cp_shift, pad, (unsigned)(row_bytes / 16));
  ctx->launches++;
  if (w) {
    niti_launch(st, (unsigned)(((long long)wrows * pitch + 255) / 256), 256, 0, widen_weights_kernel, w, ww, wrows, S, Ci, Cp, pitch);
    ctx->launches++;
  }
  NITI_CUDA_TRY(ctx, cudaGetLastError());
  return NITI_OK;
}

int niti_launch_im2col32(niti_ctx *ctx, cudaStream_t st, const int8_t *x, int8_t *xcol, int B, int H, int W,
                         int Ci, int R, int S, int pad, int stride, int Ho, int Wo) {
  if (Ci == 3 && R == 3 && S == 3 && pad == 1 && stride == 1 && (W % 4) == 0 && (long long)B * H < (1LL << 31) &&
      ((uintptr_t)xcol & 31) == 0) {
    const int threads = W / 4 >= 128 ? 128 : (W / 4 > 32 ? 64 : 32);
    const size_t smem = (size_t)3 * (W * 3 / 4 + 2) * sizeof(unsigned);
    if (smem <= 48 * 1024) {
      niti_launch(st, (unsigned)(B * H), threads, smem, im2col32_rgb3x3_kernel, x, xcol, B, H, W);
      ctx->launches++;
      NITI_CUDA_TRY(ctx, cudaGetLastError());
      return NITI_OK;
    }
  }
  long long M = (long long)B * Ho * Wo;
  long long blocks = (M + 255) / 256;
  if (blocks > (long long)ctx->sm_count * 16) blocks = (long long)ctx->sm_count * 16;
  niti_launch(st, (unsigned)blocks, 256, 0, im2col32_kernel, x, xcol, B, H, W, Ci, R, S, pad, stride, Ho, Wo);
  ctx->launches++;
  NITI_CUDA_TRY(ctx, cudaGetLastError());
  return NITI_OK;
}

int niti_launch_round_compact(niti_ctx *ctx, cudaStream_t st, const int32_t *acc, const WsHeader *hdr, int8_t *out,
                              int rows, int k, int pitch, int rowk, int rpitch, int Ci, int Cp, int mbits, int round_mode,
                              int32_t *b_out, int8_t *upd_w) {
  niti_launch(st, (rows * k + 255) / 256, 256, 0, round_compact_kernel, acc, hdr, out, rows, k, pitch, rowk, rpitch, Ci, Cp, mbits,
                                                               round_mode, b_out, upd_w);
  ctx->launches++;
  NITI_CUDA_TRY(ctx, cudaGetLastError());
  return NITI_OK;
}

// ---------------------------------------------------------------------------------------------
// Integer cross-entropy gradient, Section 3.5.  Pass 1: one warp per sample computes the integer
// T_i (Eq. 2 or Eq. 3-4), their sum, the largest magnitude of e32 = T_i - [i == label] * sum
// (64-bit) and the arg-max hit.  Pass 2: shared binary point, e32 recomputed and rounded to int8.
// ---------------------------------------------------------------------------------------------
// One warp per sample.  Pass 1 keeps two 64-bit scalars per sample (the offset p of Eq. 4 and the
// sum of the T_i) instead of the T_i themselves; pass 2 recomputes T_i from the logit, so that the only
// per-element traffic is the logit read twice and the int8 result written once.
//
// Eq. 3 in 32 bits.  x-hat of a logit is (47274 * a) >> (15 - s), a left shift when s > 15.  Without the left shift
// two different logits are already 47274 apart, more than the window of 10: every T_i is 1 with it or without it, so
// s > 15 is computed with no shift at all, and products (at most 23 bits) and thresholds fit 32 bits.  Off the label T_i
// is a power of two, at most 2^9.
constexpr int XENT_MUL = 47274;
__device__ __forceinline__ int xent_shift(int s) { return s < 15 ? 15 - s : 0; }            // (s in -6 .. 24)
__device__ __forceinline__ int xent_xhat(int a, int sh) { return (XENT_MUL * a) >> sh; }
// log2 of T_i (Eq. 4); entries above the row's largest logit are never used
__device__ __forceinline__ int xent_log_T(int a, int sh, int p) { return min(max(xent_xhat(a, sh) - p, 0), 15); }
// T_i of Eq. 2 (s <= -7)
__device__ __forceinline__ long long xent_T2(int a, int s) {
  const long long ai = a;
  return (1LL << (1 - 2 * s)) + ai * (1LL << (1 - s)) + ai * ai;
}
constexpr int XENT_WARPS = 8;

// What a row contributes: offset p of Eq. 4, sum of the T_i, largest magnitude of e32, hit.
struct XentRow {
  long long p, csum;
  unsigned long long top;
  int hit;
};
__device__ __forceinline__ bool xent_bad(int s, int label, int N) { return s < -22 || s > 24 || label < 0 || label >= N; }
__device__ __forceinline__ int hmax_s8x4(unsigned w) {
  const int b0 = (int)(int8_t)w, b1 = (int)(int8_t)(w >> 8), b2 = (int)(int8_t)(w >> 16), b3 = (int)(int8_t)(w >> 24);
  return max(max(b0, b1), max(b2, b3));
}
__device__ __forceinline__ int hmin_s8x4(unsigned w) {
  const int b0 = (int)(int8_t)w, b1 = (int)(int8_t)(w >> 8), b2 = (int)(int8_t)(w >> 16), b3 = (int)(int8_t)(w >> 24);
  return min(min(b0, b1), min(b2, b3));
}

// Units of a row: four logits (whole, aligned words) or one.  Rows of at most xent_held units per lane stay in registers
// over the sweeps of pass 1: up to 1024 logits in words, 64 as bytes.
template <bool PACKED>
constexpr int xent_held = PACKED ? 8 : 2;
template <bool PACKED>
__device__ __forceinline__ unsigned xent_unit(const int8_t *row, int i) {
  return PACKED ? reinterpret_cast<const unsigned *>(row)[i] : (unsigned)(int)row[i];
}
template <bool PACKED, bool HELD>
struct XentSweep {
  const int8_t *row;
  int units, lane;
  unsigned w[HELD ? xent_held<PACKED> : 1];
  __device__ __forceinline__ XentSweep(const int8_t *r, int n, int l) : row(r), units(n), lane(l) {
    if (HELD) {
#pragma unroll
      for (int j = 0; j < xent_held<PACKED>; ++j) {
        w[HELD ? j : 0] = 0u;
        if (lane + 32 * j < units) w[HELD ? j : 0] = xent_unit<PACKED>(row, lane + 32 * j);
      }
    }
  }
  template <typename F>
  __device__ __forceinline__ void each(F f) const {
    if (HELD) {
#pragma unroll
      for (int j = 0; j < xent_held<PACKED>; ++j)
        if (lane + 32 * j < units) f(lane + 32 * j, w[HELD ? j : 0]);
    } else {
      for (int i = lane; i < units; i += 32) f(i, xent_unit<PACKED>(row, i));
    }
  }
  // logit i of the row (the same i in the whole warp)
  __device__ __forceinline__ int logit(int i) const {
    if (!HELD) return (int)row[i];
    const int u = PACKED ? i >> 2 : i;
    unsigned x = 0;
#pragma unroll
    for (int j = 0; j < xent_held<PACKED>; ++j)
      x |= w[HELD ? j : 0] & (0u - (unsigned)(j == u >> 5));       // (masks: an index would put the words in local memory)
    x = __shfl_sync(0xffffffffu, x, u & 31);
    return PACKED ? (int)(int8_t)(x >> (8 * (i & 3))) : (int)x;
  }
};

// Pass 1 of one row by one warp.  x-hat is monotone in the logit, so a row needs: the maxima of the logits before and
// after the label (they also decide the arg-max hit), for Eq. 2 the sums of a and a^2, for Eq. 3-4 the smallest logit
// whose x-hat exceeds max - 10 (a division gives the threshold) and the sum of the powers of two.
// (s and label are in range)
template <bool PACKED, bool HELD>
__device__ __forceinline__ XentRow xent_row(const XentSweep<PACKED, HELD> &units, int N, int s, int label) {
  XentRow out;
  const int a_label = units.logit(label);
  const int lw = PACKED ? label >> 2 : label, lb = label & 3;
  int max_before = -128, max_after = -128, sum_a = 0, sum_q = 0;
  if (PACKED) {
    const unsigned low = lb == 0 ? 0u : (0xffffffffu >> (32 - 8 * lb));          // bytes before the label
    const unsigned high = lb == 3 ? 0u : (0xffffffffu << (8 * (lb + 1)));        // bytes after it
    unsigned mb = 0x80808080u, ma = 0x80808080u;
    units.each([&](int i, unsigned w) {
      sum_a = __dp4a((int)w, 0x01010101, sum_a);
      sum_q = __dp4a((int)w, (int)w, sum_q);
      const unsigned kb = i < lw ? 0xffffffffu : (i == lw ? low : 0u), ka = i > lw ? 0xffffffffu : (i == lw ? high : 0u);
      mb = __vmaxs4(mb, (w & kb) | (0x80808080u & ~kb));
      ma = __vmaxs4(ma, (w & ka) | (0x80808080u & ~ka));
    });
    max_before = hmax_s8x4(mb);
    max_after = hmax_s8x4(ma);
  } else {
    units.each([&](int i, unsigned w) {
      const int v = (int)w;
      sum_a += v;
      sum_q += v * v;
      if (i < lw) max_before = max(max_before, v);
      if (i > lw) max_after = max(max_after, v);
    });
  }
  max_before = __reduce_max_sync(0xffffffffu, max_before);
  max_after = __reduce_max_sync(0xffffffffu, max_after);
  const int max_other = max(max_before, max_after);       // -128 when the row has one element
  out.hit = (label == 0 || a_label > max_before) && a_label >= max_after ? 1 : 0;   // the first arg-max is the label
  out.p = 0;
  long long t_other, t_label;
  if (s <= -7) {
    sum_a = __reduce_add_sync(0xffffffffu, sum_a);
    sum_q = __reduce_add_sync(0xffffffffu, sum_q);
    out.csum = (long long)N * (1LL << (1 - 2 * s)) + (long long)sum_a * (1LL << (1 - s)) + (long long)sum_q;
    t_other = N > 1 ? xent_T2(max_other, s) : 0;          // T is increasing in the logit
    t_label = xent_T2(a_label, s);
  } else {
    // smallest logit value whose x-hat exceeds mx - 10: 47274 * a >= (mx - 9) * 2^sh, rounded up
    const int sh = xent_shift(s), mx = xent_xhat(max(max_other, a_label), sh);
    const int num = (mx - 9) * (1 << sh);
    const int lo = max(num > 0 ? (num + XENT_MUL - 1) / XENT_MUL : num / XENT_MUL, -128);
    // the smallest logit of the row that is at least that value
    int a_star = 127;
    if (PACKED) {
      const unsigned thr4 = (unsigned)(lo & 0xff) * 0x01010101u;
      unsigned mn = 0x7f7f7f7fu;
      units.each([&](int, unsigned w) {
        const unsigned m = __vcmpges4(w, thr4);
        mn = __vmins4(mn, (w & m) | (0x7f7f7f7fu & ~m));
      });
      a_star = hmin_s8x4(mn);
    } else {
      units.each([&](int, unsigned w) {
        if ((int)w >= lo) a_star = min(a_star, (int)w);
      });
    }
    const int p = xent_xhat(__reduce_min_sync(0xffffffffu, a_star), sh);
    int acc = 0;
    units.each([&](int, unsigned w) {
      if (PACKED) {
        acc += 1 << max(xent_xhat((int)(int8_t)w, sh) - p, 0);
        acc += 1 << max(xent_xhat((int)(int8_t)(w >> 8), sh) - p, 0);
        acc += 1 << max(xent_xhat((int)(int8_t)(w >> 16), sh) - p, 0);
        acc += 1 << max(xent_xhat((int)w >> 24, sh) - p, 0);
      } else {
        acc += 1 << max(xent_xhat((int)w, sh) - p, 0);
      }
    });
    out.p = p;
    out.csum = (long long)__reduce_add_sync(0xffffffffu, acc);
    t_other = N > 1 ? 1LL << xent_log_T(max_other, sh, p) : 0;
    t_label = 1LL << xent_log_T(a_label, sh, p);
  }
  // e32 = T_i off the label (positive) and T_label - sum (not positive) on it
  const long long on_label = out.csum - t_label;
  out.top = (unsigned long long)(t_other > on_label ? t_other : on_label);
  return out;
}

// Pass 2 of one row by one warp: off the label e32 = T(a) > 0, one rounded value per logit value, looked up in 256 bytes:
// the block's for Eq. 2 (q2), for Eq. 4 this warp's (q4), filled here from the rounded powers of two.
template <bool PACKED, bool HELD>
__device__ __forceinline__ void xent_out(const XentSweep<PACKED, HELD> &units, int8_t *__restrict__ out, int N, int s, int label, int bp,
                                         int round_mode, int p, long long csum, const unsigned char *q2, unsigned char *q4, int lane) {
  if (xent_bad(s, label, N)) {
    units.each([&](int i, unsigned) {
      if (PACKED) reinterpret_cast<unsigned *>(out)[i] = 0u;
      else out[i] = 0;
    });
    return;
  }
  const int a_label = units.logit(label), sh = xent_shift(s);
  long long t_label;
  if (s > -7) {
    // (sums of Eq. 4 are below 2^26: bp < 32)
    const unsigned q_lane = niti_round_mag<unsigned>(1u << (lane & 15), bp, 127u, round_mode);
    __syncwarp();
#pragma unroll
    for (int v = 0; v < 256; v += 32)
      q4[v + lane] = (unsigned char)__shfl_sync(0xffffffffu, q_lane, xent_log_T(v + lane - 128, sh, p));
    __syncwarp();
    t_label = 1LL << xent_log_T(a_label, sh, p);
  } else {
    t_label = xent_T2(a_label, s);
  }
  const unsigned char *q = s > -7 ? q4 : q2;
  // on the label e32 = T - sum <= 0
  const unsigned q_label =
      (unsigned)(0 - (int)niti_round_mag<unsigned long long>((unsigned long long)(csum - t_label), bp, 127ull, round_mode)) & 0xffu;
  const int lw = label >> 2, lb = label & 3;
  units.each([&](int i, unsigned v) {
    if (PACKED) {
      const unsigned w = v ^ 0x80808080u;                                  // logit + 128 per byte
      unsigned o = (unsigned)q[w & 0xff] | ((unsigned)q[(w >> 8) & 0xff] << 8) | ((unsigned)q[(w >> 16) & 0xff] << 16) |
                   ((unsigned)q[w >> 24] << 24);
      if (i == lw) o = (o & ~(0xffu << (8 * lb))) | (q_label << (8 * lb));
      reinterpret_cast<unsigned *>(out)[i] = o;
    } else {
      out[i] = (int8_t)(i == label ? q_label : (unsigned)q[(int)v + 128]);
    }
  });
}

// The rows of one block.  ONE: a single row per warp, of at most 32 * xent_held units, whose logits, offset and sum stay in
// registers between the passes; otherwise rows are strided over the warps and two scalars per row go through memory.
template <bool PACKED, bool ONE>
struct XentBlock {
  XentSweep<PACKED, ONE> held;
  XentRow mine;
  int label, blk;
  __device__ __forceinline__ static long long first_row_of(int block) {
    return (long long)block * ((int)blockDim.x >> 5) + (threadIdx.x >> 5);
  }
  __device__ __forceinline__ long long first_row() const { return first_row_of(blk); }
  __device__ __forceinline__ XentBlock(const int8_t *__restrict__ a, const int32_t *__restrict__ labels, int B, int N, int block)
      : held(a + first_row_of(block) * N, ONE && first_row_of(block) < B ? (PACKED ? N >> 2 : N) : 0, (int)threadIdx.x & 31), blk(block) {
    label = ONE && first_row() < B ? labels[first_row()] : 0;
  }
  // pass 1: the 64-bit maximum and the hits of the block, in m / h of thread 0
  __device__ __forceinline__ void stats(const int8_t *__restrict__ a, int s, const int32_t *__restrict__ labels, long long *rowinfo, int B,
                                        int N, uint32_t *status, unsigned long long *sh_max, int *sh_hit, unsigned long long &m, int &h) {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, warps = (int)blockDim.x >> 5;
    unsigned long long top = 0;
    int hits = 0;
    for (long long r = first_row(); r < B; r += (long long)gridDim.x * warps) {
      if (!ONE) label = labels[r];
      mine = {0, 0, 0ull, 0};
      if (xent_bad(s, label, N)) {
        if (lane == 0) atomicOr(status, (s < -22 || s > 24) ? NITI_DEV_XENT_RANGE : NITI_DEV_BAD_LABEL);
      } else if (ONE) {
        mine = xent_row(held, N, s, label);
      } else {
        const int units = PACKED ? N >> 2 : N;
        mine = units <= 32 * xent_held<PACKED> ? xent_row(XentSweep<PACKED, true>(a + r * N, units, lane), N, s, label)
                                       : xent_row(XentSweep<PACKED, false>(a + r * N, units, lane), N, s, label);
      }
      if (!ONE && lane == 0) {
        rowinfo[2 * r] = mine.p;
        rowinfo[2 * r + 1] = mine.csum;
      }
      top = mine.top > top ? mine.top : top;
      hits += mine.hit;
      if (ONE) break;
    }
    if (lane == 0) { sh_max[warp] = top; sh_hit[warp] = hits; }
    __syncthreads();
    m = 0;
    h = 0;
    if (threadIdx.x == 0)
      for (int w = 0; w < warps; ++w) { m = sh_max[w] > m ? sh_max[w] : m; h += sh_hit[w]; }
  }
  // pass 2.  q_tab: 256 bytes of the block, then 256 of every warp
  __device__ __forceinline__ void outs(const int8_t *__restrict__ a, int s, const int32_t *__restrict__ labels, const long long *rowinfo,
                                       int8_t *__restrict__ out, int B, int N, int bp, int round_mode, unsigned char *q_tab) {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, warps = (int)blockDim.x >> 5;
    if (s <= -7 && s >= -22) {
      if (threadIdx.x < 256)
        q_tab[threadIdx.x] =
            (unsigned char)niti_round_mag<unsigned long long>((unsigned long long)xent_T2((int)threadIdx.x - 128, s), bp, 127ull, round_mode);
      __syncthreads();
    }
    for (long long r = first_row(); r < B; r += (long long)gridDim.x * warps) {
      unsigned char *q4 = q_tab + 256 * (warp + 1);
      if (ONE) {
        xent_out(held, out + r * N, N, s, label, bp, round_mode, (int)mine.p, mine.csum, q_tab, q4, lane);
        break;
      }
      const int units = PACKED ? N >> 2 : N;
      const int p = (int)rowinfo[2 * r];
      const long long csum = rowinfo[2 * r + 1];
      if (units <= 32 * xent_held<PACKED>)
        xent_out(XentSweep<PACKED, true>(a + r * N, units, lane), out + r * N, N, s, labels[r], bp, round_mode, p, csum, q_tab, q4, lane);
      else
        xent_out(XentSweep<PACKED, false>(a + r * N, units, lane), out + r * N, N, s, labels[r], bp, round_mode, p, csum, q_tab, q4, lane);
    }
  }
};

// Both passes in two launches: the scratch has no room for an agreement (no-allocation variant), or the maximum is
// combined over the ranks in between.
template <bool PACKED>
__global__ void __launch_bounds__(32 * XENT_WARPS)
xent_row_kernel(const int8_t *__restrict__ a, const int32_t *__restrict__ s_a_ptr, const int32_t *__restrict__ labels,
                long long *rowinfo, WsHeader *hdr, int B, int N, uint32_t *__restrict__ status) {
  niti_enter(a, s_a_ptr, labels);
  __shared__ unsigned long long sh_max[XENT_WARPS];
  __shared__ int sh_hit[XENT_WARPS];
  unsigned long long m;
  int h;
  XentBlock<PACKED, false> rows(a, labels, B, N, (int)blockIdx.x);
  rows.stats(a, *s_a_ptr, labels, rowinfo, B, N, status, sh_max, sh_hit, m, h);
  if (threadIdx.x == 0) {
    if (m > *(volatile unsigned long long *)&hdr->maxabs64) atomicMax(&hdr->maxabs64, m);
    if (h) atomicAdd(&hdr->hits, (unsigned)h);
  }
}
template <bool PACKED>
__global__ void __launch_bounds__(32 * XENT_WARPS)
xent_round_kernel(const int8_t *__restrict__ a, const int32_t *__restrict__ s_a_ptr, const int32_t *__restrict__ labels,
                  const long long *rowinfo, const WsHeader *__restrict__ hdr, int8_t *__restrict__ out, int B, int N,
                  int round_mode, int32_t *__restrict__ b_out, int32_t *__restrict__ n_correct) {
  niti_enter(a, s_a_ptr, labels, rowinfo, hdr);
  __shared__ unsigned char q_tab[256 * (XENT_WARPS + 1)];
  const int b = 64 - __clzll((long long)hdr->maxabs64), bp = b > 7 ? b - 7 : 0;
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    if (b_out) *b_out = b;
    if (n_correct) *n_correct = (int32_t)hdr->hits;
  }
  XentBlock<PACKED, false> rows(a, labels, B, N, (int)blockIdx.x);
  rows.outs(a, *s_a_ptr, labels, rowinfo, out, B, N, bp, round_mode, q_tab);
}

// Both passes in one launch of at most one block per SM: the blocks agree on the bit-width in between.
// Bound: latency (a launch, one round trip for the logits, the agreement); with many rows per SM the arithmetic of pass 1.
// Two launches, of which the second reads labels, scalars and logits again, took 7.7 / 9.8 us for 64 x 1000 logits (Eq. 2 /
// Eq. 4), four with tables of all 256 offsets 13.0 / 16.8 us for 4096 x 1000 (and 29 us with their gaps outside a graph);
// one launch takes 4.7 / 5.5 and 9.2 / 11.5 us, 64 x 10 3.5 / 3.9 instead of 3.5 / 4.7 us.
constexpr int XENT_MAX_WARPS = 32;
template <bool PACKED, bool ONE, int WARPS>
__global__ void __launch_bounds__(32 * WARPS)
xent_kernel(const int8_t *__restrict__ a, const int32_t *__restrict__ s_a_ptr, const int32_t *__restrict__ labels,
            long long *rowinfo, WsHeader *hdr, int8_t *__restrict__ out, int B, int N, int round_mode, int32_t *__restrict__ b_out,
            int32_t *__restrict__ n_correct, uint32_t *__restrict__ status, unsigned patience, WsHeader *next) {
  niti_enter(a, s_a_ptr, labels);
  if (next && blockIdx.x == 0 && threadIdx.x >= 32 * (WARPS - 1)) niti_zero_header(next, (int)threadIdx.x & 31);
  __shared__ unsigned long long sh_max[WARPS];
  __shared__ int sh_hit[WARPS];
  __shared__ unsigned blk_b, grid_b, ticket;
  __shared__ unsigned char q_tab[256 * (WARPS + 1)];
  unsigned came = 0;
  if (threadIdx.x == 32 && gridDim.x > 1) came = niti_arrive(hdr);
  XentBlock<PACKED, ONE> rows(a, labels, B, N, (int)blockIdx.x);
  const int s = *s_a_ptr;
  unsigned long long m;
  int h;
  rows.stats(a, s, labels, rowinfo, B, N, status, sh_max, sh_hit, m, h);
  if (threadIdx.x == 0) {
    blk_b = 64u - (unsigned)__clzll((long long)m);
    if (gridDim.x == 1) {
      grid_b = blk_b + 1u;
      if (n_correct) *n_correct = h;
    } else if (h) {
      atomicAdd(&hdr->hits, (unsigned)h);
      __threadfence();
    }
  }
  unsigned *words = niti_split_max(hdr);
  if (gridDim.x > 1 && threadIdx.x < 32) {
    __syncwarp();
    const unsigned all = niti_agree_bits(words, words + NITI_AGREE_MAX, (int)*(volatile unsigned *)&blk_b, (int)blockIdx.x,
                                         (int)gridDim.x, 0, (int)threadIdx.x, patience);
    if (threadIdx.x == 0) grid_b = all;
  }
  if (threadIdx.x == 32) ticket = came;
  __syncthreads();
  // the scalars, by whoever rounds the first block's rows
  auto publish = [&](int b) {
    if (threadIdx.x != 0) return;
    if (b_out) *b_out = b;
    if (gridDim.x > 1 && n_correct) {                       // (every post has been seen, and thereby every hit)
      __threadfence();
      *n_correct = (int32_t)*(volatile unsigned *)&hdr->hits;
    }
  };
  const unsigned agreed = grid_b, came_as = ticket;
  if (agreed) {
    const int b = (int)agreed - 1;
    if (blockIdx.x == 0) publish(b);
    rows.outs(a, s, labels, rowinfo, out, B, N, b > 7 ? b - 7 : 0, round_mode, q_tab);
  }
  if (gridDim.x == 1 || (agreed && !(came_as >> 16))) return;
  niti_finish_left(hdr, words, agreed == 0, came_as, [&](int j) {
    const unsigned bits = niti_posted_bits(words, (int)gridDim.x, status);
    if (bits == 0) return;
    const int b = (int)bits - 1;
    if (j == 0) publish(b);
    XentBlock<PACKED, ONE> left(a, labels, B, N, j);
    if (ONE) left.stats(a, s, labels, rowinfo, B, N, status, sh_max, sh_hit, m, h);      // (the others' are in memory)
    left.outs(a, s, labels, rowinfo, out, B, N, b > 7 ? b - 7 : 0, round_mode, q_tab);
  });
}

template <bool PACKED, bool ONE>
static void launch_xent_one(int grid, int warps, cudaStream_t st, const int8_t *a, const int32_t *s_a, const int32_t *labels,
                            long long *rowinfo, WsHeader *hdr, int8_t *e, int32_t *b_e, int32_t *n_correct, int B, int N, int round_mode,
                            uint32_t *status, unsigned patience, WsHeader *next) {
  auto go = [&](auto kernel) {
    niti_launch(st, grid, 32 * warps, 0, kernel, a, s_a, labels, rowinfo, hdr, e, B, N, round_mode, b_e, n_correct, status, patience, next);
  };
  if (warps == 8) go(xent_kernel<PACKED, ONE, 8>);
  else if (warps == 16) go(xent_kernel<PACKED, ONE, 16>);
  else go(xent_kernel<PACKED, ONE, XENT_MAX_WARPS>);
}

// The packed path needs whole words per row.  (ctx may be null: the variant without a context; with one, the max
// magnitude of the 64-bit gradients is combined over the ranks between the two passes when a reduction hook is installed)
static int launch_xent(niti_ctx *ctx, cudaStream_t st, const int8_t *a, const int32_t *s_a, const int32_t *labels,
                       long long *rowinfo, WsHeader *hdr, int8_t *e, int32_t *b_e, int32_t *n_correct, int B, int N,
                       int round_mode, uint32_t *status, WsHeader *next = nullptr) {
  const bool packed = (N & 3) == 0 && N >= 64 && (((uintptr_t)a | (uintptr_t)e) & 3) == 0;
  if (ctx && !ctx->reduce_fn) {
    const int sms = ctx->sm_count < NITI_AGREE_MAX ? ctx->sm_count : NITI_AGREE_MAX;
    // few warps per block as long as there is one per row: 1024 x 1000 5.1 us with 8, 6.1 with 16, 9.9 with 32; 2048 x 100
    // 7.3 / 5.3 / 6.5 us; 4096 x 1000 13.4 / 10.6 / 9.2 us
    const int warps = B <= 8 * sms ? 8 : B <= 16 * sms ? 16 : XENT_MAX_WARPS;
    const int need = (B + warps - 1) / warps, grid = need < sms ? need : sms;
    const bool one = (packed ? N >> 2 <= 32 * xent_held<true> : N <= 32 * xent_held<false>) && B <= grid * warps;
    auto go = [&](auto launch) { launch(grid, warps, st, a, s_a, labels, rowinfo, hdr, e, b_e, n_correct, B, N, round_mode, status, ctx->patience, next); };
    if (packed) { if (one) go(launch_xent_one<true, true>); else go(launch_xent_one<true, false>); }
    else { if (one) go(launch_xent_one<false, true>); else go(launch_xent_one<false, false>); }
    ctx->launches++;
    return NITI_OK;
  }
  const unsigned blocks = (unsigned)((B + XENT_WARPS - 1) / XENT_WARPS);
  if (packed) niti_launch(st, blocks, 32 * XENT_WARPS, 0, xent_row_kernel<true>, a, s_a, labels, rowinfo, hdr, B, N, status);
  else niti_launch(st, blocks, 32 * XENT_WARPS, 0, xent_row_kernel<false>, a, s_a, labels, rowinfo, hdr, B, N, status);
  if (ctx) {
    const int rc = niti_reduce(ctx, st, &hdr->maxabs64, 1, NITI_REDUCE_MAX_U64);
    if (rc != NITI_OK) return rc;
    ctx->launches += 2;
  }
  if (packed) niti_launch(st, blocks, 32 * XENT_WARPS, 0, xent_round_kernel<true>, a, s_a, labels, rowinfo, hdr, e, B, N, round_mode, b_e, n_correct);
  else niti_launch(st, blocks, 32 * XENT_WARPS, 0, xent_round_kernel<false>, a, s_a, labels, rowinfo, hdr, e, B, N, round_mode, b_e, n_correct);
  return NITI_OK;
}

extern "C" int niti_int_xent(niti_ctx *ctx, void *stream, const int8_t *a, const int32_t *s_a,
                             const int32_t *labels, int8_t *e, int32_t *b_e, int32_t *n_correct,
                             int B, int N, int round_mode, void *ws, size_t ws_bytes) {
  if (!ctx) return NITI_ERR_ARG;
  if (!a || !s_a || !labels || !e || B <= 0 || N <= 0 || N > 65536 || (round_mode != 0 && round_mode != 1))
    return niti_fail(ctx, NITI_ERR_ARG, "niti_int_xent: bad argument");
  int64_t dims[2] = {B, N};
  if (!ws || ((uintptr_t)ws & 255) || ws_bytes < niti_workspace_bytes(NITI_OP_INT_XENT, dims, 2))
    return niti_fail(ctx, NITI_ERR_WORKSPACE, "niti_int_xent: workspace missing, misaligned or too small");
  cudaStream_t st = (cudaStream_t)stream;
  WsHeader *hdr = niti_take_header(ctx, st, ws), *next = nullptr;
  long long *rowinfo = (long long *)((char *)ws + NITI_WS_HEADER);
  const int rch = niti_clear(ctx, st, nullptr, 0, ctx->reduce_fn ? nullptr : &next);
  if (rch != NITI_OK) return rch;
  const int rcx = launch_xent(ctx, st, a, s_a, labels, rowinfo, hdr, e, b_e, n_correct, B, N, round_mode, ctx->d_status, next);
  if (rcx != NITI_OK) return rcx;
  NITI_CUDA_TRY(ctx, cudaGetLastError());
  niti_header_passed_on(ctx, next);
  return NITI_OK;
}

// ---------------------------------------------------------------------------------------------
// niti_int_xent_noalloc: the same two kernels with their scratch (reduction header + two 64-bit
// scalars per sample) in a fixed device array that is part of the library image, for callers that must
// not allocate device memory.  Every GPU that loads the library carries the array until exit.
// ---------------------------------------------------------------------------------------------
#define NITI_NOALLOC_HEADER 256       // reduction scalars of this variant (its last word: status bits)
#define NITI_NOALLOC_BYTES (NITI_NOALLOC_HEADER + 8 * NITI_XENT_NOALLOC_MAX_ELEMS)
static __device__ __align__(256) unsigned char g_xent_scratch[NITI_NOALLOC_BYTES];
// The name above is only a host-side handle in host code; the device address is looked up once per
// device (with that device current) and cached here.
static void *g_xent_scratch_addr[64];
static std::mutex g_xent_scratch_mutex;

extern "C" int niti_int_xent_noalloc(void *stream, const int8_t *a, const int32_t *s_a, const int32_t *labels,
                                     int8_t *e, int32_t *b_e, int32_t *n_correct, int B, int N, int round_mode) {
  if (!a || !s_a || !labels || !e || B <= 0 || N <= 0 || N > 65536 || (round_mode != 0 && round_mode != 1))
    return NITI_ERR_ARG;
  if ((long long)B * N > NITI_XENT_NOALLOC_MAX_ELEMS || B > NITI_XENT_NOALLOC_MAX_ELEMS / 2)
    return NITI_ERR_TOO_LARGE;                   // 16 bytes of scratch per sample must fit the array
  int dev = -1;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return NITI_ERR_CUDA;
  void *base = nullptr;
  {
    std::lock_guard<std::mutex> lock(g_xent_scratch_mutex);
    if (!g_xent_scratch_addr[dev]) {
      void *ptr = nullptr;
      if (cudaGetSymbolAddress(&ptr, g_xent_scratch) != cudaSuccess || !ptr) return NITI_ERR_CUDA;
      g_xent_scratch_addr[dev] = ptr;
    }
    base = g_xent_scratch_addr[dev];
  }
  cudaStream_t st = (cudaStream_t)stream;
  WsHeader *hdr = (WsHeader *)base;
  long long *rowinfo = (long long *)((char *)base + NITI_NOALLOC_HEADER);
  // the array keeps what the previous call left: the reduction scalars must start at zero.  The last
  // word of the header takes the (unreported) status bits of this variant.
  uint32_t *status = (uint32_t *)((char *)base + NITI_NOALLOC_HEADER - sizeof(uint32_t));
  if (cudaMemsetAsync(base, 0, NITI_NOALLOC_HEADER, st) != cudaSuccess) return NITI_ERR_CUDA;
  launch_xent(nullptr, st, a, s_a, labels, rowinfo, hdr, e, b_e, n_correct, B, N, round_mode, status);
  if (cudaGetLastError() != cudaSuccess) return NITI_ERR_CUDA;
  return NITI_OK;
}

// ---------------------------------------------------------------------------------------------
// Byte-wise SIMD elementwise ops: 16 int8 per thread per iteration (one 16-byte load per operand).
// ---------------------------------------------------------------------------------------------

__global__ void __launch_bounds__(256)
sgd_update_kernel(int8_t *__restrict__ w, const int8_t *__restrict__ g, long long n) {
  niti_enter(w, g);
  const long long nvec = n >> 4;
  const long long stride = (long long)gridDim.x * blockDim.x;
  const long long tid = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  for (long long v = tid; v < nvec; v += stride) {
    int4 wv = *(reinterpret_cast<int4 *>(w) + v);
    int4 gv = __ldcs(reinterpret_cast<const int4 *>(g) + v);
    wv.x = sat_sub_clamp127(wv.x, gv.x); wv.y = sat_sub_clamp127(wv.y, gv.y);
    wv.z = sat_sub_clamp127(wv.z, gv.z); wv.w = sat_sub_clamp127(wv.w, gv.w);
    *(reinterpret_cast<int4 *>(w) + v) = wv;
  }
  long long t = (nvec << 4) + tid;
  if (t < n) {
    int d = (int)w[t] - (int)g[t];
    d = d > 127 ? 127 : (d < -127 ? -127 : d);
    w[t] = (int8_t)d;
  }
}

__global__ void __launch_bounds__(256)
relu_fwd_kernel(const int8_t *__restrict__ x, int8_t *__restrict__ y, long long n) {
  niti_enter(x);
  const long long nvec = n >> 4;
  const long long stride = (long long)gridDim.x * blockDim.x;
  const long long tid = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  for (long long v = tid; v < nvec; v += stride) {
    int4 xv = *(reinterpret_cast<const int4 *>(x) + v);
    xv.x = __vmaxs4(xv.x, 0); xv.y = __vmaxs4(xv.y, 0); xv.z = __vmaxs4(xv.z, 0); xv.w = __vmaxs4(xv.w, 0);
    *(reinterpret_cast<int4 *>(y) + v) = xv;
  }
  long long t = (nvec << 4) + tid;
  if (t < n) y[t] = x[t] > 0 ? x[t] : 0;
}

__global__ void __launch_bounds__(256)
relu_bwd_kernel(const int8_t *__restrict__ y, const int8_t *__restrict__ eo, int8_t *__restrict__ ei,
                long long n) {
  niti_enter(y, eo);
  const long long nvec = n >> 4;
  const long long stride = (long long)gridDim.x * blockDim.x;
  const long long tid = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  for (long long v = tid; v < nvec; v += stride) {
    int4 yv = *(reinterpret_cast<const int4 *>(y) + v);
    int4 ev = *(reinterpret_cast<const int4 *>(eo) + v);
    ev.x &= __vcmpgts4(yv.x, 0); ev.y &= __vcmpgts4(yv.y, 0);
    ev.z &= __vcmpgts4(yv.z, 0); ev.w &= __vcmpgts4(yv.w, 0);
    *(reinterpret_cast<int4 *>(ei) + v) = ev;
  }
  long long t = (nvec << 4) + tid;
  if (t < n) ei[t] = y[t] > 0 ? eo[t] : 0;
}

// 2x2 max-pool, NHWC.  VEC = 16: one thread per 16 channels of one output pixel; VEC = 1: scalar.
template <int VEC>
__global__ void __launch_bounds__(256)
maxpool2_fwd_kernel(const int8_t *__restrict__ x, int8_t *__restrict__ y, int B, int H, int W, int C) {
  niti_enter(x);
  const int Ho = H >> 1, Wo = W >> 1, Cv = C / VEC;
  const long long total = (long long)B * Ho * Wo * Cv;
  for (long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x; t < total;
       t += (long long)gridDim.x * blockDim.x) {
    int cv = (int)(t % Cv);
    long long pix = t / Cv;
    int j = (int)(pix % Wo);
    long long bi = pix / Wo;
    int i = (int)(bi % Ho);
    long long b = bi / Ho;
    long long base = (((b * H + 2 * i) * W + 2 * j) * (long long)C) + (long long)cv * VEC;
    long long rs = (long long)W * C;
    if (VEC == 16) {
      int4 v0 = *reinterpret_cast<const int4 *>(x + base);
      int4 v1 = *reinterpret_cast<const int4 *>(x + base + C);
      int4 v2 = *reinterpret_cast<const int4 *>(x + base + rs);
      int4 v3 = *reinterpret_cast<const int4 *>(x + base + rs + C);
      int4 m;
      m.x = __vmaxs4(__vmaxs4(v0.x, v1.x), __vmaxs4(v2.x, v3.x));
      m.y = __vmaxs4(__vmaxs4(v0.y, v1.y), __vmaxs4(v2.y, v3.y));
      m.z = __vmaxs4(__vmaxs4(v0.z, v1.z), __vmaxs4(v2.z, v3.z));
      m.w = __vmaxs4(__vmaxs4(v0.w, v1.w), __vmaxs4(v2.w, v3.w));
      *reinterpret_cast<int4 *>(y + pix * C + (long long)cv * VEC) = m;
    } else {
      int8_t m = x[base];
      int8_t v = x[base + C]; m = v > m ? v : m;
      v = x[base + rs]; m = v > m ? v : m;
      v = x[base + rs + C]; m = v > m ? v : m;
      y[pix * C + cv] = m;
    }
  }
}

__device__ __forceinline__ void pool_bwd_word(unsigned x0, unsigned x1, unsigned x2, unsigned x3,
                                              unsigned e, int relu, unsigned &o0, unsigned &o1,
                                              unsigned &o2, unsigned &o3) {
  unsigned m = __vmaxs4(__vmaxs4(x0, x1), __vmaxs4(x2, x3));
  unsigned s0 = __vcmpeq4(x0, m);
  unsigned s1 = __vcmpeq4(x1, m) & ~s0;
  unsigned s2 = __vcmpeq4(x2, m) & ~(s0 | s1);
  unsigned s3 = ~(s0 | s1 | s2);
  if (relu) {
    unsigned pos = __vcmpgts4(m, 0);   // the routed position holds the maximum
    e &= pos;
  }
  o0 = e & s0; o1 = e & s1; o2 = e & s2; o3 = e & s3;
}

template <int VEC>
__global__ void __launch_bounds__(256)
maxpool2_bwd_kernel(const int8_t *__restrict__ x, const int8_t *__restrict__ eo,
                    int8_t *__restrict__ ei, int B, int H, int W, int C, int relu) {
  niti_enter(x, eo);
  const int Ho = H >> 1, Wo = W >> 1, Cv = C / VEC;
  const long long total = (long long)B * Ho * Wo * Cv;
  for (long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x; t < total;
       t += (long long)gridDim.x * blockDim.x) {
    int cv = (int)(t % Cv);
    long long pix = t / Cv;
    int j = (int)(pix % Wo);
    long long bi = pix / Wo;
    int i = (int)(bi % Ho);
    long long b = bi / Ho;
    long long base = (((b * H + 2 * i) * W + 2 * j) * (long long)C) + (long long)cv * VEC;
    long long rs = (long long)W * C;
    if (VEC == 16) {
      int4 v0 = *reinterpret_cast<const int4 *>(x + base);
      int4 v1 = *reinterpret_cast<const int4 *>(x + base + C);
      int4 v2 = *reinterpret_cast<const int4 *>(x + base + rs);
      int4 v3 = *reinterpret_cast<const int4 *>(x + base + rs + C);
      int4 e = *reinterpret_cast<const int4 *>(eo + pix * C + (long long)cv * VEC);
      int4 o0, o1, o2, o3;
      pool_bwd_word(v0.x, v1.x, v2.x, v3.x, e.x, relu, (unsigned &)o0.x, (unsigned &)o1.x, (unsigned &)o2.x, (unsigned &)o3.x);
      pool_bwd_word(v0.y, v1.y, v2.y, v3.y, e.y, relu, (unsigned &)o0.y, (unsigned &)o1.y, (unsigned &)o2.y, (unsigned &)o3.y);
      pool_bwd_word(v0.z, v1.z, v2.z, v3.z, e.z, relu, (unsigned &)o0.z, (unsigned &)o1.z, (unsigned &)o2.z, (unsigned &)o3.z);
      pool_bwd_word(v0.w, v1.w, v2.w, v3.w, e.w, relu, (unsigned &)o0.w, (unsigned &)o1.w, (unsigned &)o2.w, (unsigned &)o3.w);
      *reinterpret_cast<int4 *>(ei + base) = o0;
      *reinterpret_cast<int4 *>(ei + base + C) = o1;
      *reinterpret_cast<int4 *>(ei + base + rs) = o2;
      *reinterpret_cast<int4 *>(ei + base + rs + C) = o3;
    } else {
      long long idx[4] = {base, base + C, base + rs, base + rs + C};
      int best = 0;
      for (int k = 1; k < 4; ++k)
        if (x[idx[k]] > x[idx[best]]) best = k;
      int8_t e = eo[pix * C + cv];
      if (relu && x[idx[best]] <= 0) e = 0;
      for (int k = 0; k < 4; ++k) ei[idx[k]] = k == best ? e : (int8_t)0;
    }
  }
}

// ---- max-pool that records where the maximum was --------------------------------------------
// The backward pass of a 2x2 max-pool needs, per output element, the position of the first maximum
// of its window and (behind a ReLU) whether that maximum was positive: four bits.  Recording them in
// the forward pass (half a byte per output element) lets the backward pass read the error and the
// codes instead of the whole input tensor: 1.25 + 0.5/4 bytes per input element instead of 2.25.
// Code of one element: bits 0-1 = position (0: (0,0), 1: (0,1), 2: (1,0), 3: (1,1)), bit 2 = max > 0.
// Layout: [B][H/2][W/2][C/2] bytes, channel c in the low (c even) or high (c odd) nibble.
__device__ __forceinline__ unsigned pool_codes_word(unsigned x0, unsigned x1, unsigned x2, unsigned x3, unsigned &m) {
  m = __vmaxs4(__vmaxs4(x0, x1), __vmaxs4(x2, x3));
  const unsigned s0 = __vcmpeq4(x0, m);
  const unsigned s1 = __vcmpeq4(x1, m) & ~s0;
  const unsigned s2 = __vcmpeq4(x2, m) & ~(s0 | s1);
  const unsigned s3 = ~(s0 | s1 | s2);
  const unsigned pos = __vcmpgts4(m, 0);
  return (s1 & 0x01010101u) | (s2 & 0x02020202u) | (s3 & 0x03030303u) | (pos & 0x04040404u);
}
// four byte codes (one per byte) -> 16 bits of nibbles, and back
__device__ __forceinline__ unsigned pool_pack_nibbles(unsigned w) {
  const unsigned t = (w | (w >> 4)) & 0x00ff00ffu;
  return (t | (t >> 8)) & 0xffffu;
}
__device__ __forceinline__ unsigned pool_unpack_nibbles(unsigned p16) {
  const unsigned t = (p16 | (p16 << 8)) & 0x00ff00ffu;
  return (t | (t << 4)) & 0x0f0f0f0fu;
}

__global__ void __launch_bounds__(256)
maxpool2_fwd_idx_kernel(const int8_t *__restrict__ x, int8_t *__restrict__ y, uint8_t *__restrict__ idx, int B, int H,
                        int W, int C) {
  niti_enter(x);
  const int Ho = H >> 1, Wo = W >> 1, Cv = C / 16;
  const long long total = (long long)B * Ho * Wo * Cv;
  for (long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x; t < total;
       t += (long long)gridDim.x * blockDim.x) {
    const int cv = (int)(t % Cv);
    const long long pix = t / Cv;
    const int j = (int)(pix % Wo);
    const long long bi = pix / Wo;
    const int i = (int)(bi % Ho);
    const long long b = bi / Ho;
    const long long base = (((b * H + 2 * i) * W + 2 * j) * (long long)C) + (long long)cv * 16;
    const long long rs = (long long)W * C;
    const int4 v0 = *reinterpret_cast<const int4 *>(x + base);
    const int4 v1 = *reinterpret_cast<const int4 *>(x + base + C);
    const int4 v2 = *reinterpret_cast<const int4 *>(x + base + rs);
    const int4 v3 = *reinterpret_cast<const int4 *>(x + base + rs + C);
    int4 m;
    const unsigned c0 = pool_codes_word(v0.x, v1.x, v2.x, v3.x, (unsigned &)m.x);
    const unsigned c1 = pool_codes_word(v0.y, v1.y, v2.y, v3.y, (unsigned &)m.y);
    const unsigned c2 = pool_codes_word(v0.z, v1.z, v2.z, v3.z, (unsigned &)m.z);
    const unsigned c3 = pool_codes_word(v0.w, v1.w, v2.w, v3.w, (unsigned &)m.w);
    *reinterpret_cast<int4 *>(y + pix * C + (long long)cv * 16) = m;
    uint2 packed;
    packed.x = pool_pack_nibbles(c0) | (pool_pack_nibbles(c1) << 16);
    packed.y = pool_pack_nibbles(c2) | (pool_pack_nibbles(c3) << 16);
    *reinterpret_cast<uint2 *>(idx + (pix * C >> 1) + (long long)cv * 8) = packed;
  }
}

__device__ __forceinline__ void pool_route_word(unsigned codes, unsigned e, int relu, unsigned &o0, unsigned &o1,
                                                unsigned &o2, unsigned &o3) {
  const unsigned pos2 = codes & 0x03030303u;
  if (relu) e &= __vcmpne4(codes & 0x04040404u, 0u);
  o0 = e & __vcmpeq4(pos2, 0u);
  o1 = e & __vcmpeq4(pos2, 0x01010101u);
  o2 = e & __vcmpeq4(pos2, 0x02020202u);
  o3 = e & __vcmpeq4(pos2, 0x03030303u);
}

__global__ void __launch_bounds__(256)
maxpool2_bwd_idx_kernel(const int8_t *__restrict__ eo, const uint8_t *__restrict__ idx, int8_t *__restrict__ ei, int B,
                        int H, int W, int C, int relu) {
  niti_enter(eo, idx);
  const int Ho = H >> 1, Wo = W >> 1, Cv = C / 16;
  const long long total = (long long)B * Ho * Wo * Cv;
  for (long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x; t < total;
       t += (long long)gridDim.x * blockDim.x) {
    const int cv = (int)(t % Cv);
    const long long pix = t / Cv;
    const int j = (int)(pix % Wo);
    const long long bi = pix / Wo;
    const int i = (int)(bi % Ho);
    const long long b = bi / Ho;
    const long long base = (((b * H + 2 * i) * W + 2 * j) * (long long)C) + (long long)cv * 16;
    const long long rs = (long long)W * C;
    const int4 e = __ldcs(reinterpret_cast<const int4 *>(eo + pix * C + (long long)cv * 16));
    const uint2 packed = __ldcs(reinterpret_cast<const uint2 *>(idx + (pix * C >> 1) + (long long)cv * 8));
    int4 o0, o1, o2, o3;
    pool_route_word(pool_unpack_nibbles(packed.x & 0xffffu), e.x, relu, (unsigned &)o0.x, (unsigned &)o1.x, (unsigned &)o2.x, (unsigned &)o3.x);
    pool_route_word(pool_unpack_nibbles(packed.x >> 16), e.y, relu, (unsigned &)o0.y, (unsigned &)o1.y, (unsigned &)o2.y, (unsigned &)o3.y);
    pool_route_word(pool_unpack_nibbles(packed.y & 0xffffu), e.z, relu, (unsigned &)o0.z, (unsigned &)o1.z, (unsigned &)o2.z, (unsigned &)o3.z);
    pool_route_word(pool_unpack_nibbles(packed.y >> 16), e.w, relu, (unsigned &)o0.w, (unsigned &)o1.w, (unsigned &)o2.w, (unsigned &)o3.w);
    *reinterpret_cast<int4 *>(ei + base) = o0;
    *reinterpret_cast<int4 *>(ei + base + C) = o1;
    *reinterpret_cast<int4 *>(ei + base + rs) = o2;
    *reinterpret_cast<int4 *>(ei + base + rs + C) = o3;
  }
}

static inline unsigned ew_blocks(niti_ctx *ctx, long long work_items) {
  long long blocks = (work_items + 255) / 256;
  long long cap = (long long)ctx->sm_count * 16;
  if (blocks > cap) blocks = cap;
  if (blocks < 1) blocks = 1;
  return (unsigned)blocks;
}

int niti_launch_sgd_update(niti_ctx *ctx, cudaStream_t st, int8_t *w, const int8_t *g, long long n) {
  niti_launch(st, ew_blocks(ctx, (n >> 4) + 16), 256, 0, sgd_update_kernel, w, g, n);
  ctx->launches++;
  NITI_CUDA_TRY(ctx, cudaGetLastError());
  return NITI_OK;
}

extern "C" int niti_int_sgd_update(niti_ctx *ctx, void *stream, int8_t *w, const int8_t *g, int64_t n) {
  if (!ctx) return NITI_ERR_ARG;
  if (!w || !g || n <= 0) return niti_fail(ctx, NITI_ERR_ARG, "niti_int_sgd_update: bad argument");
  if (((uintptr_t)w | (uintptr_t)g) & 15)
    return niti_fail(ctx, NITI_ERR_ARG, "niti_int_sgd_update: pointers must be 16-byte aligned");
  niti_launch((cudaStream_t)stream, ew_blocks(ctx, (n >> 4) + 16), 256, 0, sgd_update_kernel, w, g, n);
  ctx->launches++;
  NITI_CUDA_TRY(ctx, cudaGetLastError());
  return NITI_OK;
}

// Several tensors copied by one launch (bound: memory).  A block copies 32 KB of one tensor; blocks find their tensor by
// a search over the (at most 32) first blocks.  The sixteen weight tensors of the VGG-16 stack took 60 us as sixteen
// copies, most of them 1.5 - 2 us each for a few KB.
constexpr int COPY_MAX = 32;
constexpr int COPY_BLOCK_BYTES = 32768;
struct CopyList {
  int8_t *dst[COPY_MAX];
  const int8_t *src[COPY_MAX];
  long long bytes[COPY_MAX];
  int first[COPY_MAX + 1];        // first block of each tensor
  int n;
};
__global__ void __launch_bounds__(256)
copy_many_kernel(const __grid_constant__ CopyList l) {
  niti_enter();
  int t = 0;
  while (t + 1 < l.n && (int)blockIdx.x >= l.first[t + 1]) ++t;
  const long long off = (long long)((int)blockIdx.x - l.first[t]) * COPY_BLOCK_BYTES;
  const int left = l.bytes[t] - off < COPY_BLOCK_BYTES ? (int)(l.bytes[t] - off) : COPY_BLOCK_BYTES;
  const int8_t *src = l.src[t] + off;
  int8_t *dst = l.dst[t] + off;
  const int nv = left >> 4;
  if (nv == COPY_BLOCK_BYTES / 16) {
    uint4 v[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) v[i] = __ldcs(reinterpret_cast<const uint4 *>(src) + threadIdx.x + 256 * i);
#pragma unroll
    for (int i = 0; i < 8; ++i) reinterpret_cast<uint4 *>(dst)[threadIdx.x + 256 * i] = v[i];
  } else {
    for (int i = threadIdx.x; i < nv; i += 256) reinterpret_cast<uint4 *>(dst)[i] = reinterpret_cast<const uint4 *>(src)[i];
    for (int i = 16 * nv + threadIdx.x; i < left; i += 256) dst[i] = src[i];
  }
}

extern "C" int niti_copy_tensors(niti_ctx *ctx, void *stream, int n, void *const *dst, const void *const *src,
                                 const int64_t *bytes) {
  if (!ctx) return NITI_ERR_ARG;
  if (n < 0 || (n > 0 && (!dst || !src || !bytes))) return niti_fail(ctx, NITI_ERR_ARG, "niti_copy_tensors: bad argument");
  for (int i = 0; i < n; ++i)
    if (!dst[i] || !src[i] || bytes[i] < 0 || bytes[i] > (1LL << 43) || (((uintptr_t)dst[i] | (uintptr_t)src[i]) & 15))
      return niti_fail(ctx, NITI_ERR_ARG, "niti_copy_tensors: bad argument (tensors must be 16-byte aligned)");
  for (int i0 = 0; i0 < n; i0 += COPY_MAX) {
    CopyList l;
    l.n = n - i0 < COPY_MAX ? n - i0 : COPY_MAX;
    long long blocks = 0;
    for (int i = 0; i < l.n; ++i) {
      l.dst[i] = (int8_t *)dst[i0 + i];
      l.src[i] = (const int8_t *)src[i0 + i];
      l.bytes[i] = bytes[i0 + i];
      l.first[i] = (int)blocks;
      blocks += (l.bytes[i] + COPY_BLOCK_BYTES - 1) / COPY_BLOCK_BYTES;
    }
    l.first[l.n] = (int)blocks;
    if (blocks >= (1LL << 31)) return niti_fail(ctx, NITI_ERR_SHAPE, "niti_copy_tensors: too many bytes");
    if (!blocks) continue;
    niti_launch((cudaStream_t)stream, (unsigned)blocks, 256, 0, copy_many_kernel, l);
    ctx->launches++;
    NITI_CUDA_TRY(ctx, cudaGetLastError());
  }
  return NITI_OK;
}

extern "C" int niti_relu_fwd(niti_ctx *ctx, void *stream, const int8_t *x, int8_t *y, int64_t n) {
  if (!ctx) return NITI_ERR_ARG;
  if (!x || !y || n <= 0 || (((uintptr_t)x | (uintptr_t)y) & 15))
    return niti_fail(ctx, NITI_ERR_ARG, "niti_relu_fwd: bad argument");
  niti_launch((cudaStream_t)stream, ew_blocks(ctx, (n >> 4) + 16), 256, 0, relu_fwd_kernel, x, y, n);
  ctx->launches++;
  NITI_CUDA_TRY(ctx, cudaGetLastError());
  return NITI_OK;
}

extern "C" int niti_relu_bwd(niti_ctx *ctx, void *stream, const int8_t *y, const int8_t *e_out,
                             int8_t *e_in, int64_t n) {
  if (!ctx) return NITI_ERR_ARG;
  if (!y || !e_out || !e_in || n <= 0 || (((uintptr_t)y | (uintptr_t)e_out | (uintptr_t)e_in) & 15))
    return niti_fail(ctx, NITI_ERR_ARG, "niti_relu_bwd: bad argument");
  niti_launch((cudaStream_t)stream, ew_blocks(ctx, (n >> 4) + 16), 256, 0, relu_bwd_kernel, y, e_out, e_in, n);
  ctx->launches++;
  NITI_CUDA_TRY(ctx, cudaGetLastError());
  return NITI_OK;
}

int niti_launch_maxpool2_fwd(niti_ctx *ctx, cudaStream_t st, const int8_t *x, int8_t *y, int B, int H, int W, int C) {
  bool vec = (C % 16 == 0) && !(((uintptr_t)x | (uintptr_t)y) & 15);
  long long items = (long long)B * (H / 2) * (W / 2) * (vec ? C / 16 : C);
  if (vec)
    niti_launch(st, ew_blocks(ctx, items), 256, 0, maxpool2_fwd_kernel<16>, x, y, B, H, W, C);
  else
    niti_launch(st, ew_blocks(ctx, items), 256, 0, maxpool2_fwd_kernel<1>, x, y, B, H, W, C);
  ctx->launches++;
  NITI_CUDA_TRY(ctx, cudaGetLastError());
  return NITI_OK;
}

extern "C" int niti_maxpool2_fwd(niti_ctx *ctx, void *stream, const int8_t *x, int8_t *y, int B, int H,
                                 int W, int C) {
  if (!ctx) return NITI_ERR_ARG;
  if (!x || !y || B <= 0 || H <= 0 || W <= 0 || C <= 0 || (H & 1) || (W & 1))
    return niti_fail(ctx, NITI_ERR_ARG, "niti_maxpool2_fwd: bad argument (H and W must be even)");
  return niti_launch_maxpool2_fwd(ctx, (cudaStream_t)stream, x, y, B, H, W, C);
}

extern "C" int niti_maxpool2_fwd_idx(niti_ctx *ctx, void *stream, const int8_t *x, int8_t *y, uint8_t *idx, int B,
                                     int H, int W, int C) {
  if (!ctx) return NITI_ERR_ARG;
  if (!x || !y || !idx || B <= 0 || H <= 0 || W <= 0 || C <= 0 || (H & 1) || (W & 1))
    return niti_fail(ctx, NITI_ERR_ARG, "niti_maxpool2_fwd_idx: bad argument (H and W must be even)");
  if ((C % 16) != 0 || (((uintptr_t)x | (uintptr_t)y) & 15) || ((uintptr_t)idx & 7))
    return niti_fail(ctx, NITI_ERR_SHAPE, "niti_maxpool2_fwd_idx: C must be a multiple of 16 and the tensors aligned");
  const long long items = (long long)B * (H / 2) * (W / 2) * (C / 16);
  niti_launch((cudaStream_t)stream, ew_blocks(ctx, items), 256, 0, maxpool2_fwd_idx_kernel, x, y, idx, B, H, W, C);
  ctx->launches++;
  NITI_CUDA_TRY(ctx, cudaGetLastError());
  return NITI_OK;
}

extern "C" int niti_maxpool2_bwd_idx(niti_ctx *ctx, void *stream, const int8_t *e_out, const uint8_t *idx,
                                     int8_t *e_in, int B, int H, int W, int C, int relu) {
  if (!ctx) return NITI_ERR_ARG;
  if (!e_out || !idx || !e_in || B <= 0 || H <= 0 || W <= 0 || C <= 0 || (H & 1) || (W & 1))
    return niti_fail(ctx, NITI_ERR_ARG, "niti_maxpool2_bwd_idx: bad argument (H and W must be even)");
  if ((C % 16) != 0 || (((uintptr_t)e_out | (uintptr_t)e_in) & 15) || ((uintptr_t)idx & 7))
    return niti_fail(ctx, NITI_ERR_SHAPE, "niti_maxpool2_bwd_idx: C must be a multiple of 16 and the tensors aligned");
  const long long items = (long long)B * (H / 2) * (W / 2) * (C / 16);
  niti_launch((cudaStream_t)stream, ew_blocks(ctx, items), 256, 0, maxpool2_bwd_idx_kernel, e_out, idx, e_in, B, H, W, C, relu);
  ctx->launches++;
  NITI_CUDA_TRY(ctx, cudaGetLastError());
  return NITI_OK;
}

extern "C" int niti_maxpool2_bwd(niti_ctx *ctx, void *stream, const int8_t *x, const int8_t *e_out,
                                 int8_t *e_in, int B, int H, int W, int C, int relu) {
  if (!ctx) return NITI_ERR_ARG;
  if (!x || !e_out || !e_in || B <= 0 || H <= 0 || W <= 0 || C <= 0 || (H & 1) || (W & 1))
    return niti_fail(ctx, NITI_ERR_ARG, "niti_maxpool2_bwd: bad argument (H and W must be even)");
  bool vec = (C % 16 == 0) && !(((uintptr_t)x | (uintptr_t)e_out | (uintptr_t)e_in) & 15);
  long long items = (long long)B * (H / 2) * (W / 2) * (vec ? C / 16 : C);
  if (vec)
    niti_launch((cudaStream_t)stream, ew_blocks(ctx, items), 256, 0, maxpool2_bwd_kernel<16>, x, e_out, e_in, B, H, W, C, relu);
  else
    niti_launch((cudaStream_t)stream, ew_blocks(ctx, items), 256, 0, maxpool2_bwd_kernel<1>, x, e_out, e_in, B, H, W, C, relu);
  ctx->launches++;
  NITI_CUDA_TRY(ctx, cudaGetLastError());
  return NITI_OK;
}
