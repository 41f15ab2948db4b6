// Small fully connected multiplies (at most NITI_SMALL_MACS multiply-accumulates): one launch that loads, multiplies,
// agrees on the bit-width, rounds and stores; a backward call runs its error and weight-gradient multiplies in the
// same launch.
//
// Bound: latency.  On the tcgen05 kernel a 64 x 256 x 784 layer took 10 - 13 us of which the multiply is a few hundred
// nanoseconds: tensor-memory allocation, barriers and descriptors (1.3 us), first TMA data (2.8 us), tensor-memory
// round trips.  Here a CTA copies its operands with asynchronous copies issued at once, multiplies with mma.sync
// (m16n8k32, int8) from shared memory, and the CTAs (at most one per SM) exchange their maxima through words of the
// workspace header.  (One cluster of up to 16 CTAs that exchanges them through distributed shared memory measured the
// same at 4 M multiply-accumulates, 5.4 against 5.2 us, and slower above, 8.2 against 5.8 us at 256^3.)
// Measured (graph replay, forward / backward call, other kernels -> this): 256 x 10 x 512 9.0 / 36.0 -> 6.6 / 8.0 us, 512 x 512
// x 256 8.6 / 18.3 -> 7.0 / 12.0, 512 x 512 x 512 9.4 / 18.5 -> 8.7 / 14.2, 512 x 512 x 700 13.0 / 24.0 -> 11.9 / 15.2, 64 x
// 1024 x 2048 12.3 / 20.0 -> 10.1 / 20.2.
// The line at NITI_SMALL_MACS: at 134 - 185 M multiply-accumulates as above; at 268 M 10.4 - 10.6 -> 10.1 - 10.3 us forward and
// 19.1 - 24.1 -> 16.8 - 24.0 us backward, about even; at 537 M 10.8 / 21.0 - 23.4 -> 11.9 - 12.1 / 23.4 - 27.9 us.
//
// Contraction order.  mma.sync wants k = 4t .. 4t+3 and 16 + 4t .. from thread t of a group; any permutation of k that
// both operands share gives the same sums, so a thread takes the 16 contiguous bytes at 16 t of a 64-byte step: one
// 16-byte shared load per row feeds two MMAs.  Rows are permuted too: fragment row g of the four 8-row groups of a
// 32 x 32 warp tile is matrix row 4g + group, which makes a thread's results 8 contiguous columns.
#include "niti_common.cuh"

namespace {

constexpr int SMALL_THREADS = 512;
constexpr int SMALL_WARPS = SMALL_THREADS / 32;
constexpr size_t SMALL_SMEM = 200 * 1024;

// One multiply out[m][n] = sum_k A(m, k) B(n, k).  An operand is K-major (row r, element k at p[r * ld + k]) or
// MN-major (p[k * ld + r]).
struct SmallOp {
  const int8_t *a, *b;
  int lda, ldb;
  int gm, gn, gk;
  int rm, rn, cn;             // region of a CTA (multiples of 32), CTAs per row of regions
  int ctas;                   // CTAs of this multiply (0: this launch has no such multiply)
  int kc;                     // contraction elements staged at a time (multiple of 64)
  int a_mn, b_mn, mbits, relu;
  int8_t *out;
  const int8_t *mask;         // output is zero where mask <= 0
  int8_t *upd;                // weights from which the rounded result is subtracted (out is then not written)
  const int32_t *s_a, *s_w;
  int32_t *s_out, *b_out;
};
struct SmallParams {
  SmallOp op[2];              // op[0]: forward or error; op[1]: the weight gradient beside an error
  int round_mode;
  unsigned patience;
  WsHeader *hdr;              // cleared
  WsHeader *next;             // to be cleared for the next call, or null
  int32_t *left;              // in the workspace: sums of regions whose CTAs left, [gm][gn] of op[0], then of op[1]
  uint32_t *status;
};

__device__ __forceinline__ unsigned smem_addr(const void *p) { return (unsigned)__cvta_generic_to_shared(p); }
// asynchronous copy of SIZE bytes, those from the `bytes`-th on zero
template <int SIZE>
__device__ __forceinline__ void cp_async(unsigned dst, const void *src, int bytes) {
  if (SIZE == 16) asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(bytes) : "memory");
  else asm volatile("cp.async.ca.shared.global [%0], [%1], %2, %3;" ::"r"(dst), "l"(src), "n"(SIZE), "r"(bytes) : "memory");
}
template <int SIZE>
__device__ __forceinline__ void stage_rows(const int8_t *p, int ld, int gk, int r0, int rv, int k0, int kc, int8_t *dst) {
  const int parts = kc / SIZE;
  for (int idx = threadIdx.x; idx < rv * parts; idx += SMALL_THREADS) {
    const int r = idx / parts, c = (idx - r * parts) * SIZE;
    int n = gk - k0 - c;
    n = n < 0 ? 0 : (n > SIZE ? SIZE : n);
    const int8_t *src = p + (long long)(r0 + r) * ld + k0 + (n > 0 ? c : 0);
    cp_async<SIZE>(smem_addr(dst + r * (kc + 16) + c), src, n);
  }
}
__device__ __forceinline__ void mma_s8(int (&c)[4], const unsigned (&a)[4], unsigned b0, unsigned b1) {
  asm volatile("mma.sync.aligned.m16n8k32.row.col.s32.s8.s8.s32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};"
               : "+r"(c[0]), "+r"(c[1]), "+r"(c[2]), "+r"(c[3])
               : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
// Stages rows r0 .. r0 + rows - 1, elements k0 .. k0 + kc - 1 of an operand as dst[row][kc + 16], zero beyond gk.
// Rows beyond the matrix are left as they are (their results are never used).
__device__ __forceinline__ void stage_operand(const int8_t *p, int ld, int mn, int extent, int gk, int r0, int rows, int k0,
                                              int kc, int8_t *dst) {
  const int pitch = kc + 16;
  const int rv = extent - r0 < rows ? extent - r0 : rows;          // rows inside the matrix
  if (!mn) {
    const unsigned al = (unsigned)ld | (unsigned)(uintptr_t)p;
    if ((al & 15) == 0) {
      stage_rows<16>(p, ld, gk, r0, rv, k0, kc, dst);
    } else if ((al & 7) == 0) {
      stage_rows<8>(p, ld, gk, r0, rv, k0, kc, dst);
    } else if ((al & 3) == 0) {
      stage_rows<4>(p, ld, gk, r0, rv, k0, kc, dst);
    } else {
      // rows at any byte: words through registers, eight in flight per thread
      const int words = kc >> 2, total = rv * words;
      for (int base = threadIdx.x; base < total; base += 8 * SMALL_THREADS) {
        unsigned v[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) {
          const int idx = base + u * SMALL_THREADS;
          const int r = idx / words, c = (idx - r * words) * 4;
          v[u] = idx < total ? niti_load_bytes4(p + (long long)(r0 + r) * ld + k0 + c, gk - k0 - c) : 0u;
        }
#pragma unroll
        for (int u = 0; u < 8; ++u) {
          const int idx = base + u * SMALL_THREADS;
          const int r = idx / words, c = (idx - r * words) * 4;
          if (idx < total) *reinterpret_cast<unsigned *>(dst + r * pitch + c) = v[u];
        }
      }
    }
    return;
  }
  // 4 x 4 byte blocks, transposed on the way; a warp takes 16 blocks along k and 2 along the rows (conflict-free stores)
  const int rq_n = (rv + 3) >> 2, rq2 = (rq_n + 1) >> 1, kq16 = kc >> 6;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const bool words_ok = (ld & 3) == 0 && ((uintptr_t)p & 3) == 0;
  constexpr int UNR = 4;                                            // blocks in flight per thread
  for (int job0 = warp; job0 < rq2 * kq16; job0 += UNR * SMALL_WARPS) {
    unsigned w[UNR][4];
#pragma unroll
    for (int u = 0; u < UNR; ++u) {
      const int job = job0 + u * SMALL_WARPS;
      const int jr = job / kq16, jk = job - jr * kq16;
      const int rq = jr * 2 + (lane >> 4), k = (jk * 16 + (lane & 15)) * 4;
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        w[u][i] = 0u;
        if (rq < rq_n && k0 + k + i < gk) {
          const int8_t *src = p + (long long)(k0 + k + i) * ld + r0 + 4 * rq;
          w[u][i] = words_ok && 4 * rq + 4 <= rv ? *reinterpret_cast<const unsigned *>(src) : niti_load_bytes4(src, rv - 4 * rq);
        }
      }
    }
#pragma unroll
    for (int u = 0; u < UNR; ++u) {
      const int job = job0 + u * SMALL_WARPS;
      const int jr = job / kq16, jk = job - jr * kq16;
      const int rq = jr * 2 + (lane >> 4), k = (jk * 16 + (lane & 15)) * 4;
      if (rq >= rq_n) continue;
      const unsigned t0 = __byte_perm(w[u][0], w[u][1], 0x5140), t1 = __byte_perm(w[u][2], w[u][3], 0x5140);
      const unsigned t2 = __byte_perm(w[u][0], w[u][1], 0x7362), t3 = __byte_perm(w[u][2], w[u][3], 0x7362);
      int8_t *d = dst + (4 * rq) * pitch + k;
      *reinterpret_cast<unsigned *>(d) = __byte_perm(t0, t1, 0x5410);
      *reinterpret_cast<unsigned *>(d + pitch) = __byte_perm(t0, t1, 0x7632);
      *reinterpret_cast<unsigned *>(d + 2 * pitch) = __byte_perm(t2, t3, 0x5410);
      *reinterpret_cast<unsigned *>(d + 3 * pitch) = __byte_perm(t2, t3, 0x7632);
    }
  }
}

// Rounds and stores the region at (m0, n0), of CTA c of its multiply, whose sums are in shared memory.
__device__ __forceinline__ void round_region(const SmallParams &p, const SmallOp &o, const int *acc, int c, int m0, int n0,
                                             unsigned agreed_bits) {
  const int tid = threadIdx.x, acc_pitch = o.rn + 4;
  const int b = (int)agreed_bits - 1, bp = b > o.mbits ? b - o.mbits : 0;
  const unsigned qmax = (1u << o.mbits) - 1u;
  if (c == 0 && tid == 0) {
    if (o.b_out) *o.b_out = b;
    if (o.s_out) {
      const int s = bp + (o.s_a ? *o.s_a : 0) + (o.s_w ? *o.s_w : 0);
      *o.s_out = s;
      if (s < -128 || s > 127) atomicOr(p.status, NITI_DEV_EXP_RANGE);
    }
  }
  const int q = o.rn >> 2;
  int8_t *dst = o.upd ? o.upd : o.out;
  const bool words_ok = (o.gn & 3) == 0 && (((uintptr_t)dst | (uintptr_t)o.mask) & 3) == 0;
  for (int idx = tid; idx < o.rm * q; idx += SMALL_THREADS) {
    const int r = idx / q, cc = (idx - r * q) * 4;
    const int nv = o.gn - n0 - cc;
    if (m0 + r >= o.gm || nv <= 0) continue;
    const long long off = (long long)(m0 + r) * o.gn + n0 + cc;
    const int4 v = *reinterpret_cast<const int4 *>(acc + r * acc_pitch + cc);
    const int xs[4] = {v.x, v.y, v.z, v.w};
    unsigned w = 0;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      int x = niti_round_i32(xs[j], bp, qmax, p.round_mode);
      if (o.relu && x < 0) x = 0;
      w |= (unsigned)(x & 0xff) << (8 * j);
    }
    if (words_ok) {
      if (o.mask) w &= __vcmpgts4(*reinterpret_cast<const unsigned *>(o.mask + off), 0u);
      if (o.upd) w = __vmaxs4(__vsubss4(*reinterpret_cast<const unsigned *>(dst + off), w), 0x81818181u);
      *reinterpret_cast<unsigned *>(dst + off) = w;
    } else {
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        if (j >= nv) break;
        int x = (int)(int8_t)(w >> (8 * j));
        if (o.mask && o.mask[off + j] <= 0) x = 0;
        if (o.upd) {
          x = (int)dst[off + j] - x;
          x = x > 127 ? 127 : (x < -127 ? -127 : x);
        }
        dst[off + j] = (int8_t)x;
      }
    }
  }
}
__device__ __forceinline__ int32_t *left_sums(const SmallParams &p, int which) {
  return p.left + (which ? (long long)p.op[0].gm * p.op[0].gn : 0);
}
// The regions of CTAs that left (see niti_agree_bits).
__device__ __forceinline__ void finish_left_regions(const SmallParams &p, int *acc, bool left, unsigned ticket) {
  unsigned *words = niti_split_max(p.hdr);
  const int ctas0 = p.op[0].ctas;
  niti_finish_left(p.hdr, words, left, ticket, [&](int j) {
    const int which = (j < ctas0 || p.op[1].ctas == 0) ? 0 : 1;
    const SmallOp &o = p.op[which];
    const int c = which ? j - ctas0 : j, m0 = c / o.cn * o.rm, n0 = c % o.cn * o.rn;
    const unsigned bits = niti_posted_bits(words + (which ? ctas0 : 0), o.ctas, p.status);
    if (bits == 0 || (which && o.upd && niti_posted_bits(words, ctas0, p.status) == 0)) return;      // (op[0] reads the weights)
    __threadfence();
    __syncthreads();
    const int32_t *sums = left_sums(p, which);
    for (int idx = threadIdx.x; idx < o.rm * o.rn; idx += SMALL_THREADS) {
      const int r = idx / o.rn, cc = idx - r * o.rn;
      if (m0 + r < o.gm && n0 + cc < o.gn) acc[r * (o.rn + 4) + cc] = __ldcg(sums + (long long)(m0 + r) * o.gn + n0 + cc);
    }
    __syncthreads();
    round_region(p, o, acc, c, m0, n0, bits);
  });
}

__global__ void __launch_bounds__(SMALL_THREADS, 1)
small_gemm_kernel(const __grid_constant__ SmallParams p) {
  extern __shared__ __align__(16) int8_t smem[];
  __shared__ unsigned cta_max, agreed, ticket;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  // which multiply, which region
  const int ctas0 = p.op[0].ctas;
  const int which = ((int)blockIdx.x < ctas0 || p.op[1].ctas == 0) ? 0 : 1;
  const SmallOp &o = p.op[which];
  const int first = which ? ctas0 : 0;
  const int cta = (int)blockIdx.x - first;
  const int cm_i = cta / o.cn, cn_i = cta - cm_i * o.cn;
  const int m0 = cm_i * o.rm, n0 = cn_i * o.rn;
  const int acc_pitch = o.rn + 4;
  int *acc = reinterpret_cast<int *>(smem);                 // [rm][rn + 4]
  int8_t *As = smem + (size_t)o.rm * acc_pitch * 4, *Bs = As + o.rm * (o.kc + 16);
  if (tid == 0) cta_max = 0;
  niti_enter();
  unsigned came = 0;
  if (blockIdx.x == 0 && warp == SMALL_WARPS - 1 && p.next) niti_zero_header(p.next, lane);
  if (tid == 32) came = niti_arrive(p.hdr);
  unsigned mx = 0;
  {
    const int tiles_n = o.rn >> 5, tiles = (o.rm >> 5) * tiles_n;
    const int steps_c = o.kc >> 6;                          // 64-element steps of a full chunk
    int wk = SMALL_WARPS / tiles;                           // warps that share a tile along k
    wk = wk < 1 ? 1 : (wk > steps_c ? steps_c : wk);
    const bool direct = wk == 1 && o.kc >= o.gk;            // one writer per result
    if (!direct)
      for (int i = tid; i < o.rm * acc_pitch; i += SMALL_THREADS) acc[i] = 0;
    for (int k0 = 0; k0 < o.gk; k0 += o.kc) {
      if (k0) __syncthreads();                              // the previous chunk has been read
      stage_operand(o.a, o.lda, o.a_mn, o.gm, o.gk, m0, o.rm, k0, o.kc, As);
      stage_operand(o.b, o.ldb, o.b_mn, o.gn, o.gk, n0, o.rn, k0, o.kc, Bs);
      asm volatile("cp.async.commit_group;\n\tcp.async.wait_group 0;" ::: "memory");
      __syncthreads();
      const int left = o.gk - k0, steps = left >= o.kc ? steps_c : (left + 63) >> 6;
      const int per = (steps + wk - 1) / wk, pitch = o.kc + 16;
      const int g = lane >> 2, t = lane & 3;
      for (int job = warp; job < tiles * wk; job += SMALL_WARPS) {
        const int tile = job / wk, ks = job - tile * wk;
        const int tm = tile / tiles_n, tn = tile - tm * tiles_n;
        const int s0 = ks * per, s1 = s0 + per < steps ? s0 + per : steps;
        int c[2][4][4];
#pragma unroll
        for (int i = 0; i < 2; ++i)
#pragma unroll
          for (int j = 0; j < 4; ++j)
#pragma unroll
            for (int q = 0; q < 4; ++q) c[i][j][q] = 0;
        const int8_t *ap = As + (tm * 32 + 4 * g) * pitch + 16 * t, *bp = Bs + (tn * 32 + 4 * g) * pitch + 16 * t;
        for (int s = s0; s < s1; ++s) {
          uint4 av[4], bv[4];
#pragma unroll
          for (int r = 0; r < 4; ++r) {
            av[r] = *reinterpret_cast<const uint4 *>(ap + r * pitch + 64 * s);
            bv[r] = *reinterpret_cast<const uint4 *>(bp + r * pitch + 64 * s);
          }
#pragma unroll
          for (int i = 0; i < 2; ++i) {
            const unsigned a0[4] = {av[2 * i].x, av[2 * i + 1].x, av[2 * i].y, av[2 * i + 1].y};
            const unsigned a1[4] = {av[2 * i].z, av[2 * i + 1].z, av[2 * i].w, av[2 * i + 1].w};
#pragma unroll
            for (int j = 0; j < 4; ++j) {
              mma_s8(c[i][j], a0, bv[j].x, bv[j].y);
              mma_s8(c[i][j], a1, bv[j].z, bv[j].w);
            }
          }
        }
        // rows 4g + 2i (+ 1), columns 8t + j and 8t + 4 + j
#pragma unroll
        for (int i = 0; i < 2; ++i)
#pragma unroll
          for (int h = 0; h < 2; ++h) {
            int *row = acc + (tm * 32 + 4 * g + 2 * i + h) * acc_pitch + tn * 32 + 8 * t;
            if (direct) {
              *reinterpret_cast<int4 *>(row) = make_int4(c[i][0][2 * h], c[i][1][2 * h], c[i][2][2 * h], c[i][3][2 * h]);
              *reinterpret_cast<int4 *>(row + 4) =
                  make_int4(c[i][0][2 * h + 1], c[i][1][2 * h + 1], c[i][2][2 * h + 1], c[i][3][2 * h + 1]);
            } else if (s0 < s1) {
#pragma unroll
              for (int j = 0; j < 4; ++j) {
                atomicAdd(row + j, c[i][j][2 * h]);
                atomicAdd(row + 4 + j, c[i][j][2 * h + 1]);
              }
            }
          }
      }
    }
    __syncthreads();
    // largest magnitude of the region
    const int q = o.rn >> 2;
    for (int idx = tid; idx < o.rm * q; idx += SMALL_THREADS) {
      const int r = idx / q, cc = (idx - r * q) * 4;
      if (m0 + r >= o.gm) continue;
      const int4 v = *reinterpret_cast<const int4 *>(acc + r * acc_pitch + cc);
      const int nv = o.gn - n0 - cc;
      if (nv > 0) mx = max(mx, (unsigned)abs(v.x));
      if (nv > 1) mx = max(mx, (unsigned)abs(v.y));
      if (nv > 2) mx = max(mx, (unsigned)abs(v.z));
      if (nv > 3) mx = max(mx, (unsigned)abs(v.w));
    }
  }
  mx = __reduce_max_sync(0xffffffffu, mx);
  if (lane == 0 && mx) atomicMax(&cta_max, mx);
  __syncthreads();
  // agreement over the CTAs of this multiply.  The exchange also orders the weight update of op[1] after op[0]'s reads of
  // the same weights: an update waits for op[0]'s CTAs as well.  (Those reads have returned, into shared memory and behind a
  // barrier, before op[0] posts, and a write issued after the post was seen cannot reach a read that has returned.  Fences or
  // acquiring loads on top of that cost a captured MLP step 43.4 -> 45.1 - 46.0 us.)
  if (warp == 0) {
    unsigned *words = niti_split_max(p.hdr);
    const unsigned m = niti_agree_bits(words + first, words + NITI_AGREE_MAX + 4 * first, niti_bitlen32(cta_max), cta, o.ctas,
                                       o.upd ? first : 0, lane, p.patience);
    if (lane == 0) agreed = m;
  }
  if (tid == 32) ticket = came;
  __syncthreads();
  const unsigned bits = agreed, came_as = ticket;
  if (bits) {
    round_region(p, o, acc, cta, m0, n0, bits);
  } else {
    int32_t *sums = left_sums(p, which);
    for (int idx = tid; idx < o.rm * o.rn; idx += SMALL_THREADS) {
      const int r = idx / o.rn, c = idx - r * o.rn;
      if (m0 + r < o.gm && n0 + c < o.gn) sums[(long long)(m0 + r) * o.gn + n0 + c] = acc[r * acc_pitch + c];
    }
  }
  if (bits == 0 || came_as >> 16) finish_left_regions(p, acc, bits == 0, came_as);
}

inline int up32(long long v) { return (int)((v + 31) / 32 * 32); }
inline size_t region_smem(int rm, int rn, int kc) { return (size_t)rm * (rn + 4) * 4 + (size_t)(rm + rn) * (kc + 16); }

// Regions of one multiply over at most `max_ctas` CTAs: the split with the least modelled time of a CTA (operand bytes
// at about 32 per clock, 512 multiply-accumulates and two results per clock).  False when no region fits.
bool pick_regions(SmallOp &o, int max_ctas) {
  double best = 1e30;
  for (int cm = 1; cm <= max_ctas && (cm - 1) * 32 < o.gm; ++cm) {
    const int rm = up32((o.gm + cm - 1) / cm);
    const int cn = max_ctas / ((o.gm + rm - 1) / rm);
    if (cn < 1) continue;
    const int rn = up32((o.gn + cn - 1) / cn);
    if ((long long)rm * rn > 24576) continue;
    int kc = (o.gk + 63) / 64 * 64;
    while (kc > 64 && region_smem(rm, rn, kc) > SMALL_SMEM) kc = (kc / 2 + 63) / 64 * 64;
    if (region_smem(rm, rn, kc) > SMALL_SMEM) continue;
    const double t = (double)(rm + rn) * o.gk / 32 + (double)rm * rn * o.gk / 512 + (double)rm * rn / 2;
    if (t < best * 0.999) {
      best = t;
      o.rm = rm; o.rn = rn; o.kc = kc;
      o.cn = (o.gn + rn - 1) / rn;
      o.ctas = (o.gm + rm - 1) / rm * o.cn;
    }
  }
  return best < 1e30;
}

// Staging that the tcgen05 kernel beats, whatever the number of multiply-accumulates.  (1) A contraction that does not fit
// shared memory in one piece: the pieces are loaded one after the other, and the regions are few (forward 64 x 128 x 9216 25.6
// against 9.7 us, 256 x 100 x 4096 15.6 / 10.5, 96 x 512 x 4000 15.5 / 11.4; backward 20000 x 64 x 64 128 / 24, 8192 x 128 x
// 128 59 / 21, 4096 x 128 x 256 33 / 23; in one piece 64 x 1024 x 2600 13.0 / 17.2, 3000 x 300 x 200 23.6 / 30.7).  (2) Rows
// that begin at any byte, which go through registers at about 0.125 us per KB: 1000 x 500 x 370 (47 KB per CTA) 15.6 / 12.8
// us, 500 x 300 x 999 (96 KB) 21.3 / 14.9, with 368 and 992 elements 9.4 / 10.7 and 9.9 / 11.2.
constexpr long long SMALL_ANY_BYTE = 24 * 1024;
bool slow_staging(const SmallOp &o) {
  const long long rows = (!o.a_mn && (o.lda & 3) ? o.rm : 0) + (!o.b_mn && (o.ldb & 3) ? o.rn : 0);
  return o.kc < o.gk || rows * o.gk > SMALL_ANY_BYTE;
}
// Beside the CUDA-core engine (backward, fewer than 32 outputs) pieces still pay up to this contraction: gradient of 8192 x 10 x
// 9216 90 against 503 us, 2048 x 31 x 4096 20 / 225, 4096 x 10 x 1024 28 / 101, 16384 x 10 x 1024 96 / 105, 32768 x 10 x 1024
// 186 / 200, but 65536 x 10 x 784 360 / 276.
constexpr long long SMALL_NARROW_K = 32768;

}  // namespace

static void fill_op(SmallOp &o, const GemmProblem &g, const RoundSpec &r) {
  memset(&o, 0, sizeof(o));
  o.a = g.p0; o.b = g.p1;
  o.gm = (int)g.gm; o.gn = (int)g.gn; o.gk = (int)g.gk;
  o.lda = g.kind == GK_FC_FWD ? g.K : g.N;
  o.ldb = g.K;
  o.a_mn = g.kind == GK_FC_WGRAD;
  o.b_mn = g.kind != GK_FC_FWD;
  o.out = r.out; o.mask = r.mask; o.upd = r.update_w;
  o.mbits = r.mbits; o.relu = r.relu ? 1 : 0;
  o.s_a = r.s_a; o.s_w = r.s_w; o.s_out = r.s_out; o.b_out = r.b_out;
}

// Runs one multiply (g2 == null) or the two multiplies of a backward call in one launch.  NITI_ERR_SHAPE: not a
// small problem, nothing was enqueued.
int niti_small_gemm(niti_ctx *ctx, cudaStream_t st, void *ws, const GemmProblem &g, const RoundSpec &r,
                    const GemmProblem *g2, const RoundSpec *r2) {
  const double macs = (double)g.M * g.N * g.K;
  const bool narrow = g.N < 32 && g.kind != GK_FC_FWD;             // (the alternative is the CUDA-core engine)
  if (ctx->engine != 0 || ctx->reduce_fn || g.kind > GK_FC_WGRAD || macs > NITI_SMALL_MACS * (narrow ? NITI_SMALL_NARROW : 1) || g.gk > NITI_SPLIT_MAX_K ||
      (g2 && g2->gk > NITI_SPLIT_MAX_K))
    return NITI_ERR_SHAPE;
  SmallParams p;
  memset(&p, 0, sizeof(p));
  p.round_mode = r.round_mode;
  p.status = ctx->d_status;
  fill_op(p.op[0], g, r);
  if (g2) fill_op(p.op[1], *g2, *r2);
  if (!ctx->small_ready) {
    NITI_CUDA_TRY(ctx, cudaFuncSetAttribute(small_gemm_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)SMALL_SMEM));
    ctx->small_ready = 1;
  }
  const int n = ctx->sm_count < NITI_AGREE_MAX ? ctx->sm_count : NITI_AGREE_MAX;
  if (!pick_regions(p.op[0], g2 ? n / 2 : n)) return NITI_ERR_SHAPE;
  if (g2 && !pick_regions(p.op[1], n - p.op[0].ctas)) return NITI_ERR_SHAPE;
  if (narrow ? g.gk > SMALL_NARROW_K || (g2 && g2->gk > SMALL_NARROW_K) : slow_staging(p.op[0]) || (g2 && slow_staging(p.op[1])))
    return NITI_ERR_SHAPE;
  const int grid = p.op[0].ctas + p.op[1].ctas;
  size_t smem = region_smem(p.op[0].rm, p.op[0].rn, p.op[0].kc);
  if (g2) {
    const size_t s2 = region_smem(p.op[1].rm, p.op[1].rn, p.op[1].kc);
    if (s2 > smem) smem = s2;
  }
  WsHeader *hdr = niti_take_header(ctx, st, ws);
  const int rc = niti_clear(ctx, st, nullptr, 0, &p.next);
  if (rc != NITI_OK) return rc;
  p.hdr = hdr;
  p.patience = ctx->patience;
  p.left = (int32_t *)((char *)ws + NITI_WS_HEADER);
  NITI_CUDA_TRY(ctx, niti_launch(st, (unsigned)grid, SMALL_THREADS, smem, small_gemm_kernel, p));
  niti_header_passed_on(ctx, p.next);
  ctx->launches++;
  ctx->tc_launches += g2 ? 2 : 1;
  return NITI_OK;
}
