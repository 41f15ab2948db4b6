// Tensor-core engine: int8 x int8 -> int32 matrix multiply on the 5th-generation tensor cores
// (tcgen05.mma kind::i8, accumulators in tensor memory, operands staged by TMA), sm_100a only.
//
// One persistent CTA (or CTA pair) per SM, 20 warps: warps 0..2 = TMA producers (each owns every
// third stage of the ring), warp 3 = MMA issuer and TMEM owner, warps 4..19 = epilogue (four per
// 32-lane quarter of TMEM, read with tcgen05.ld).  Up to eight accumulator buffers live in TMEM, so
// the epilogues of finished tiles overlap the main loops of the following ones.
//
// The six operand mappings of the layer ops (Int8MatrixMultiply of Algorithm 1; implicit GEMM for
// convolutions, Section 3.2) differ only in the TMA tensor maps, the per-k-block coordinates the
// producer issues, and the shared-memory matrix descriptors (K-major or MN-major operands).
//
// Every wait in the kernel is bounded: after ~1 s without progress a thread raises
// NITI_DEV_TIMEOUT in the status word, and all roles drain and leave through the common exit
// that frees the tensor memory.
#include "niti_common.cuh"
#include "niti_div.h"
#include <math.h>
#include <type_traits>

namespace {

constexpr int BM = 128;               // rows of an output tile = TMEM lanes
constexpr int EPI_WARPS = 16;          // four per TMEM lane quarter, interleaved 32-column chunks
constexpr int EPI_PER_Q = EPI_WARPS / 4;
// TMA copies are issued by single threads, and one thread sustains only about one copy per
// 250 ns (measured: four issuing warps give four times the copy rate), so the k-blocks are dealt
// round-robin to PROD_WARPS producer warps.
constexpr int PROD_WARPS = 3;          // each stage of the ring belongs to one producer warp (stage % nprod)
constexpr int MMA_WARP = PROD_WARPS;
constexpr int EPI_WARP0 = PROD_WARPS + 1;
constexpr int NUM_THREADS = 32 * (PROD_WARPS + 1 + EPI_WARPS);
constexpr int MAX_STAGES = 8;
constexpr int MAX_TBUF = 8;
constexpr long long WAIT_LIMIT_CYCLES = 2000000000LL;

// What the fused epilogue does with a launch's tiles; one instance of its loop each.
enum LeanForm {
  LEAN_PLAIN = 0, LEAN_RELU, LEAN_MASK, LEAN_POOL, LEAN_UPDATE,
  LEAN_NARROW, LEAN_NARROW_RELU, LEAN_NARROW_MASK,                   // output rows that are not whole, aligned 32-byte chunks
  LEAN_BATCHED, LEAN_BATCHED_RELU, LEAN_BATCHED_NARROW, LEAN_BATCHED_NARROW_RELU     // row-batched items
};
// How a tile's rows lie in the output
enum RowKind { ROWS_HALO = 0, ROWS_BOXES, ROWS_PLAIN, ROWS_PHASES, ROWS_WGRAD };

struct TcParams {
  int kind;
  int form, row_kind;           // LeanForm, RowKind
  int io_unit;                  // 32: output (and mask) rows are whole, aligned chunks; else the largest store unit, at most 16
  Div d_w, d_h;                 // w_tiles, h_tiles
  Div d_n, d_split;             // n_tiles_n, splits
  Div d_group, d_units, d_last; // rasterisation: tiles of a group, its row units, those of the last group
  int last_group;
  Div d_chunks, d_S, d_cc;      // n_chunks, S, c_chunks
  Div d_phases, d_phase_s;      // nph_r * nph_s, nph_s
  int wt_shift, ht_shift;       // log2 of Wt, Ht (pixel boxes)
  int k_wpq_shift;              // log2 of k_wpq
  int n_tiles_n;                // tiles along the output columns
  int kb_total;                 // k-blocks of the whole contraction
  int kb_per_split;
  int splits;
  long long items;              // tiles * splits
  // set-up arithmetic done on the host (integer divisions at kernel entry delay every launch)
  int blk_per, blk_extra;       // blocked assignment: items per CTA (pair) and how many take one more
  int k_wpq, k_wpq_active, k_epi_active, k_tmem_cols;
  unsigned patience;            // cycles that CTAs wait for each other
  int nissue;                   // resident-weights mode: warps that issue MMAs (2: the warp that loaded the
                                // weights takes every other tile)
  int one_commit;               // resident-weights mode with as many patch stages as accumulator buffers:
                                // stage and buffer advance together, one barrier per tile serves both
  int red;                      // split contraction whose partial sums are added by TMA reduce copies (map_c)
  int red_off;                  // byte offset (from the aligned base) of the epilogue warps' 4 KB buffers for them
  int nstg_off;                 // byte offset of the staging buffers for rows with a pitch that is no multiple of 8
  int mrep;                     // 128-row tiles per item (row-batched mode of short contractions), else 1
  int bn_mma;                   // N of one MMA; bn = mrep * bn_mma accumulator columns per item
  int gm, gn;                   // output extent (rows, columns; gm * gn < 2^31); row pitch of acc is gn
  int bn;                       // tile width (multiple of 32, <= 256)
  int kdepth;                   // contraction elements per k-block (32, 64 or 128)
  int ksteps;                   // kdepth / 32 MMAs per k-block
  int stages;
  // shared-memory layout of one stage
  int a_bytes, b_bytes;         // bytes of the A and B parts of a stage
  int a_boxes, b_boxes;         // TMA copies per operand per stage
  int a_box_bytes, b_box_bytes;
  int a_box_step, b_box_step;   // coordinate step between consecutive boxes (MN-major operands)
  // MMA descriptors
  unsigned idesc;
  unsigned long long a_desc, b_desc;   // descriptor without the start address
  unsigned a_kstep16, b_kstep16;       // start-address advance per MMA, in 16-byte units
  // convolution geometry (pixels of the tensor that the 4-D map covers)
  int Wt, Ht, Bt;               // pixel box of a tile / k-block: Wt * Ht * Bt == 128
  int w_tiles, h_tiles, b_tiles;
  int PW, PH, PB;               // extent of the pixel grid the output rows (or k-blocks) run over
  int R, S, pad;
  int stride_w;                 // the same for columns (1 where the input is a tensor of windows)
  int stride;                   // convolution stride (forward and weight gradient; the shifted operand is then
                                // copied with that element stride, so a box still lands as Wt x Ht pixels)
  int c_chunks;                 // channel chunks per tap along the contraction (fwd / dgrad)
  int tail_ks;                  // MMAs of the last channel chunk when it is not a whole one (0: all chunks whole)
  // im2col copies (see "Pixel rows" at the planner): rows / contraction pixels are consecutive pixels of the
  // PB x PH x PW grid, whatever its extents
  int mode;                     // kernel instance: see "Instances" at the kernel
  int i2c;
  int i2c_w0, i2c_h0;           // base pixel (in the copied tensor) of grid position (0, 0)
  int i2c_dj, i2c_di, i2c_db;   // wgrad: 128 pixels as (columns, rows, images) of the grid
  // error of a strided convolution: dstride > 1.  Input pixels with the same (position + pad) mod stride form a
  // phase, whose error is a stride-1 correlation of e with every dstride-th tap; items run over (tile, phase)
  int dstride;
  int nph_r, nph_s;             // phases with at least one tap
  int T_r, T_s;                 // taps of the phase with most of them
  int u0_r, u0_s;               // first grid position: input row = dstride * (position + u0) + phase - pad
  int OH, OW;                   // extent of the tensor the output rows are written to
  int Cn;                       // wgrad: input channels Ci (columns per tap)
  int n_chunks;                 // wgrad: column chunks per tap
  int tg, tg_cols, tg_boxes;    // wgrad: taps per column tile (tap groups), columns and copies (per CTA) of one tap
  int ctas;                     // CTAs per tile: 1, or 2 (cta_group::2, 256-row tiles)
  int m_units;                  // row units: 128-row tiles (ctas = 1) or 256-row pairs (ctas = 2)
  int raster_g;                 // row units per rasterisation group (0: row-major order)
  int blocked;                  // 1: every CTA takes a contiguous range of items (its first tile then
                                //    samples the tensor evenly), 0: items strided over the grid
  int nbuf;                     // accumulator buffers in tensor memory (2..8)
  int egroups;                  // epilogue warp groups (1, 2 or 4); tile `use` belongs to group use % egroups
  int nprod;                    // producer warps in use; divides `stages` (each stage has one owner, so
                                // the waits on a stage's barriers stay in order)
  // halo mode (3x3 convolutions with few channels): the weights of all nine taps stay in shared
  // memory for the whole kernel, every tile loads its 8 x 16 pixel patch once with a one-pixel
  // halo (10 x 18 pixels), and the nine taps are nine row offsets into that patch
  // halo == 2: weight gradient of such a convolution for one (64 output channels, 64 input
  // channels) block.  Per 8 x 16 pixel tile the CTA loads the error tile and the input patch once;
  // the nine taps are row offsets into the patch, two taps share one MMA (M = 2 x 64 input
  // channels through the leading-dimension stride of the MN-major descriptor), N = 64 output
  // channels, and the five accumulators stay in tensor memory over the CTA's whole pixel range.
  int halo;
  int wg_nci;                   // 64-channel blocks of the input channels
  int b_tile_bytes;             // bytes of one tap's weight tile
  int b_res_bytes;              // bytes of the resident weights (all taps), multiple of 1024
  int b_resident;               // generic loops: the B tiles of all k-blocks (b_tile_bytes each) stay in shared memory as well
  // epilogue
  int epi_mode;                 // EPI_SPILL / EPI_ATOMIC / EPI_SPECULATE / EPI_KNOWN_B
  int mbits, round_mode, relu;
  unsigned spec_mul256;         // the sampled max is scaled by this / 256 before taking its bit length
  unsigned trial_mul256;        // the same for the maximum of a CTA's own first tile (see lean_as), 0: no trial
  int spec_tag;                 // identifies the call site (its b_out scalar) in the table of estimate errors
  int update;                   // 1: out8 holds weights: the epilogue stores clamp(w - rounded gradient, +-127)
  int pool;                     // 1: the epilogue also stores the 2 x 2 max-pool of the (ReLU'd) output tile
  int pool_xh;                  // lane distance of the pixel one image row below (the pixel to the right is lane ^ 1)
  WsHeader *next;               // header to be zeroed for the next call, or null
  int single_wave;              // every CTA has at most one tile: the sample is the whole tensor, the shift
                                // is exact, and whoever rounds the first CTA's tile publishes b and the exponent
};

// Epilogue modes.  The shift of Algorithm 2 needs the bit-width of the WHOLE accumulator tensor:
//  EPI_SPILL      store int32 accumulators + max; a second kernel rounds (always exact, 8 B / output
//                 of extra traffic)
//  EPI_ATOMIC     split contraction: add partial sums into a zeroed int32 tensor, 32 x 32 values per TMA reduce copy.
//                 (An SM retires only about 1.6 atomic additions per cycle from registers, 4.9 us for a 64 x 256 tile
//                 and 11 us for a 128 x 256 one; the reduce copies add at L2 in whole lines.)
//  EPI_SPECULATE  every CTA computes its first tile, the grid agrees on the max over those tiles
//                 (one bounded grid-wide wait), and all tiles are rounded and stored as int8 with the
//                 shift that max implies, while the true max is tracked.  Unless every CTA has used
//                 exactly the true bit-width, the EPI_KNOWN_B pass recomputes everything with it (exact in
//                 all cases; the common case costs one multiply and no int32 traffic)
//  EPI_KNOWN_B    bit-width known (hdr->maxabs32): round and store directly.  The kernel returns at
//                 once when the speculative pass was right.
enum { EPI_SPILL = 0, EPI_ATOMIC = 1, EPI_SPECULATE = 2, EPI_KNOWN_B = 3 };


// ------------------------------------------------------------------------------------------
// PTX wrappers
// ------------------------------------------------------------------------------------------
__device__ __forceinline__ unsigned smem_u32(const void *p) {
  return (unsigned)__cvta_generic_to_shared(p);
}
__device__ __forceinline__ void mbar_init(unsigned bar, unsigned count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count));
}
__device__ __forceinline__ void mbar_expect_tx(unsigned bar, unsigned bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ void mbar_arrive(unsigned bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ bool mbar_try(unsigned bar, unsigned parity) {
  unsigned ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(bar), "r"(parity)
      : "memory");
  return ok != 0;
}
// Same, but the thread may sleep in hardware for up to `ns` nanoseconds while the phase is pending
// (it is woken when the phase completes), so a waiting warp does not burn issue slots polling.
__device__ __forceinline__ bool mbar_try_sleep(unsigned bar, unsigned parity, unsigned ns) {
  unsigned ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(bar), "r"(parity), "r"(ns)
      : "memory");
  return ok != 0;
}
// A waiting warp that keeps polling takes issue slots next to the working warps of its scheduler (the
// hardware wait above returns after a few tens of cycles: ncu counts a poll loop every ~70 cycles in a
// warp that waits through an epilogue-bound tile).  After two failed polls the warp sleeps between
// polls, 128 ns at first and 256 ns from the eighth poll on.  Run times with and without the sleep
// measured the same within 1 % on five layer shapes; the sleep is kept because it costs nothing and
// leaves the issue slots to the working warps.
__device__ __forceinline__ void wait_backoff(unsigned &polls) {
  ++polls;
  if (polls > 2) __nanosleep(polls > 8 ? 256u : 128u);
}
// Bounded wait.  Returns false (and raises the abort flag) if the barrier did not flip in time or
// another thread already gave up.
__device__ __forceinline__ bool mbar_wait(unsigned bar, unsigned parity, volatile int *abort_flag,
                                          uint32_t *status, long long limit_cycles = WAIT_LIMIT_CYCLES) {
  if (mbar_try(bar, parity)) return true;
  long long t0 = clock64();
  unsigned polls = 0;
  while (true) {
    if (mbar_try_sleep(bar, parity, 20000u)) return true;
    if (*abort_flag) return false;
    if (clock64() - t0 > limit_cycles) {
      *abort_flag = 1;
      atomicOr(status, NITI_DEV_TIMEOUT);
      return false;
    }
    wait_backoff(polls);
  }
}
// The same bounded wait for a whole converged warp: every lane polls, the votes make the outcome (and
// with it the caller's control flow) warp-uniform, so the compiler can keep the caller's address
// arithmetic in uniform registers.
__device__ __forceinline__ bool mbar_wait_warp(unsigned bar, unsigned parity, volatile int *abort_flag,
                                               uint32_t *status, long long limit_cycles = WAIT_LIMIT_CYCLES) {
  if (__all_sync(0xffffffffu, mbar_try(bar, parity))) return true;
  const long long t0 = clock64();
  unsigned polls = 0;
  while (true) {
    if (__all_sync(0xffffffffu, mbar_try_sleep(bar, parity, 20000u))) return true;
    if (__any_sync(0xffffffffu, *abort_flag != 0)) return false;
    if (__any_sync(0xffffffffu, clock64() - t0 > limit_cycles)) {
      *abort_flag = 1;
      atomicOr(status, NITI_DEV_TIMEOUT);
      return false;
    }
    wait_backoff(polls);
  }
}
// One lane of a converged warp (the same one every time it is asked).
__device__ __forceinline__ bool elect_one() {
  unsigned pred;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "elect.sync _|p, 0xffffffff;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(pred));
  return pred != 0;
}
__device__ __forceinline__ void tma_load_2d(unsigned dst, const CUtensorMap *map, unsigned bar, int c0, int c1) {
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4}], [%2];"
      ::"r"(dst), "l"(map), "r"(bar), "r"(c0), "r"(c1)
      : "memory");
}
__device__ __forceinline__ void tma_load_4d(unsigned dst, const CUtensorMap *map, unsigned bar, int c0, int c1,
                                            int c2, int c3) {
  asm volatile(
      "cp.async.bulk.tensor.4d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, %5, %6}], [%2];"
      ::"r"(dst), "l"(map), "r"(bar), "r"(c0), "r"(c1), "r"(c2), "r"(c3)
      : "memory");
}
__device__ __forceinline__ void tma_load_3d(unsigned dst, const CUtensorMap *map, unsigned bar, int c0, int c1, int c2) {
  asm volatile(
      "cp.async.bulk.tensor.3d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, %5}], [%2];"
      ::"r"(dst), "l"(map), "r"(bar), "r"(c0), "r"(c1), "r"(c2)
      : "memory");
}
// im2col copy of consecutive pixels: base pixel (w, h, n), filter offset (ow, oh)
__device__ __forceinline__ void tma_load_im2col(unsigned dst, const CUtensorMap *map, unsigned bar, int c, int w, int h,
                                                int n, unsigned short ow, unsigned short oh) {
  asm volatile(
      "cp.async.bulk.tensor.4d.shared::cluster.global.im2col.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, %5, %6}], [%2], {%7, %8};"
      ::"r"(dst), "l"(map), "r"(bar), "r"(c), "r"(w), "r"(h), "r"(n), "h"(ow), "h"(oh)
      : "memory");
}
// Adds a 32 x 32 int32 tile from shared memory (rows of 128 bytes, 128-byte swizzle) into the accumulator tensor;
// elements outside the tensor are left out.
__device__ __forceinline__ void tma_reduce_add_4d(const CUtensorMap *map, unsigned src, int c0, int c1, int c2, int c3) {
  asm volatile(
      "cp.reduce.async.bulk.tensor.4d.global.shared::cta.add.tile.bulk_group [%0, {%2, %3, %4, %5}], [%1];\n\t"
      "cp.async.bulk.commit_group;"
      ::"l"(map), "r"(src), "r"(c0), "r"(c1), "r"(c2), "r"(c3)
      : "memory");
}
// this thread's reduce copies have read their source / are complete
__device__ __forceinline__ void tma_reduce_wait_read() { asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory"); }
__device__ __forceinline__ void tma_reduce_wait_all() { asm volatile("cp.async.bulk.wait_group 0;" ::: "memory"); }
__device__ __forceinline__ void fence_async_shared() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }
__device__ __forceinline__ void st_shared_v4(unsigned addr, int a, int b, int c, int d) {
  asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(addr), "r"(a), "r"(b), "r"(c), "r"(d) : "memory");
}
__device__ __forceinline__ void st_shared_b32(unsigned addr, int a) {
  asm volatile("st.shared.b32 [%0], %1;" ::"r"(addr), "r"(a) : "memory");
}
// One lane's 32 values as row `lane` (or, TRANSPOSED, as column `lane`) of the swizzled tile at `buf`.
template <bool TRANSPOSED>
__device__ __forceinline__ void stage_tile32(unsigned buf, int lane, const int (&v)[32]) {
  if (TRANSPOSED) {
#pragma unroll
    for (int j = 0; j < 32; ++j)
      st_shared_b32(buf + (unsigned)(j * 128 + ((((lane >> 2) ^ (j & 7)) << 4) | ((lane & 3) << 2))), v[j]);
  } else {
#pragma unroll
    for (int j = 0; j < 8; ++j)
      st_shared_v4(buf + (unsigned)(lane * 128 + ((j ^ (lane & 7)) << 4)), v[4 * j], v[4 * j + 1], v[4 * j + 2], v[4 * j + 3]);
  }
}
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_commit(unsigned bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}
// Same with the two 64-bit matrix descriptors given as 32-bit halves: the issuing thread then does
// its address arithmetic in 32 bits (the high halves never change inside a kernel).
__device__ __forceinline__ void tc_mma_i8_lh(unsigned tmem_d, unsigned a_lo, unsigned a_hi, unsigned b_lo,
                                             unsigned b_hi, unsigned idesc, unsigned accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t.reg .b64 da, db;\n\t"
      "setp.ne.b32 p, %6, 0;\n\t"
      "mov.b64 da, {%1, %2};\n\t"
      "mov.b64 db, {%3, %4};\n\t"
      "tcgen05.mma.cta_group::1.kind::i8 [%0], da, db, %5, p;\n\t}"
      ::"r"(tmem_d), "r"(a_lo), "r"(a_hi), "r"(b_lo), "r"(b_hi), "r"(idesc), "r"(accumulate)
      : "memory");
}
__device__ __forceinline__ void tc_ld32(unsigned taddr, int (&v)[32]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
      "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
      "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
      : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]),
        "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15]),
        "=r"(v[16]), "=r"(v[17]), "=r"(v[18]), "=r"(v[19]), "=r"(v[20]), "=r"(v[21]), "=r"(v[22]), "=r"(v[23]),
        "=r"(v[24]), "=r"(v[25]), "=r"(v[26]), "=r"(v[27]), "=r"(v[28]), "=r"(v[29]), "=r"(v[30]), "=r"(v[31])
      : "r"(taddr)
      : "memory");
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
}

// Shift-and-round of four accumulators (Algorithm 2 + 3, or round-to-nearest) packed into four int8.
//
// Pseudo-stochastic rule on a magnitude a with bp discarded bits (h = bp / 2, o = bp & 1): the lowest
// bit is dropped when bp is odd; the next 2h bits are top * 2^h + bot and the integer part is
// incremented iff top > bot.  With mask2 = (2^h - 1) << o the term (~a & mask2) is (2^h - 1 - bot) << o,
// and adding it times 2^h carries into bit bp exactly when top > bot:
//     q = (a + (~a & mask2) * 2^h) >> bp           (the dropped lowest bit cannot carry).
// Round-to-nearest is the same expression with mask2 = 0 and the constant 2^(bp-1) in place of the
// product.  Saturation at 2^mbits - 1 happens only when the integer part is already 2^mbits - 1, so
// clamping the magnitude to cap = (2^mbits - 1) << bp beforehand gives the same result.
//
// The integer pipe of an SM issues one warp instruction every two cycles, and the epilogue of every
// output element runs on it: the instruction count per element here bounds the layers with few
// input channels.  ReLU outputs therefore never form |x|: max(min(x, cap), 0) is one instruction and
// rounds negative inputs to zero by itself; the true extremes are tracked with three-input min/max.
struct RoundConst {
  unsigned mask2;   // (2^h - 1) << o, or 0
  unsigned orc;     // 0, or 1 for round-to-nearest with bp > 0
  unsigned mulp;    // 2^h, or 2^(bp-1)
  int shift;        // bp
  int cap;          // (2^mbits - 1) << bp
  unsigned hi_mul;  // 2^(32 - bp) for bp > 0: the high half of v * hi_mul is v >> bp
  // Byte-aligned form (bp <= 24): with k = (8 - bp % 8) % 8 the sum scaled by 2^k has its integer
  // part exactly in byte B = (bp + k) / 8, so no shift is needed: a byte permute picks the rounded
  // values of two accumulators at once.
  unsigned sc;      // 2^k
  unsigned c2;      // mulp * 2^k
  unsigned sel;     // permute selector: byte B of either operand in bytes 0 and 1, zeros above
  unsigned m16;     // 2^16 (merges two byte pairs with a multiply-add)
  bool aligned;
};
__device__ __forceinline__ RoundConst make_round_const(int bp, int mbits, int round_mode) {
  RoundConst k;
  k.shift = bp;
  k.cap = (int)(((1u << mbits) - 1u) << bp);
  k.hi_mul = bp > 0 ? 1u << (32 - bp) : 0u;
  if (round_mode == NITI_ROUND_PSR) {
    const int h = bp >> 1;
    k.mask2 = ((1u << h) - 1u) << (bp & 1);
    k.orc = 0;
    k.mulp = 1u << h;
  } else {
    k.mask2 = 0;
    k.orc = bp > 0 ? 1u : 0u;
    k.mulp = bp > 0 ? 1u << (bp - 1) : 0u;
  }
  const int kk = (8 - (bp & 7)) & 7, B = (bp + kk) >> 3;
  k.aligned = bp <= 24;
  k.sc = 1u << kk;
  k.c2 = k.mulp << kk;
  // (kept opaque: known to be a power of two, the multiplies would be turned back into shifts on
  // the integer pipe, which is the one that has no slots to spare)
  k.m16 = 0x10000u;
  asm volatile("" : "+r"(k.sc), "+r"(k.c2), "+r"(k.m16));
  // selector nibbles: B (first operand), 4 + B (second operand), then twice "sign of byte B"
  // replicated, which is zero because a rounded magnitude is at most 127
  k.sel = (unsigned)B | ((unsigned)(4 + B) << 4) | ((unsigned)(8 | B) << 8) | ((unsigned)(8 | B) << 12);
  return k;
}
// magnitude already clamped to cap
template <bool SHIFT>
__device__ __forceinline__ unsigned round_mag1(unsigned m, const RoundConst &k) {
  const unsigned v = (((~m) & k.mask2) | k.orc) * k.mulp + m;
  return SHIFT ? __umulhi(v, k.hi_mul) : v;
}
// Extremes of the raw accumulators seen by one thread.
struct Extremes {
  int hi, lo;       // running max (>= 0) and min (<= 0)
  unsigned orv;     // OR of magnitudes (same bit length as their maximum)
  __device__ __forceinline__ unsigned magnitude_bits() const {
    return orv | (unsigned)hi | (0u - (unsigned)lo);
  }
};
template <bool RELU, bool SHIFT>
__device__ __forceinline__ unsigned round_pack4(int x0, int x1, int x2, int x3, const RoundConst &k, Extremes &e) {
  unsigned q0, q1, q2, q3;
  if (RELU) {
    e.hi = __vimax3_s32(e.hi, x0, x1);
    e.hi = __vimax3_s32(e.hi, x2, x3);
    e.lo = __vimin3_s32(e.lo, x0, x1);
    e.lo = __vimin3_s32(e.lo, x2, x3);
    q0 = round_mag1<SHIFT>((unsigned)__vimin_s32_relu(x0, k.cap), k);
    q1 = round_mag1<SHIFT>((unsigned)__vimin_s32_relu(x1, k.cap), k);
    q2 = round_mag1<SHIFT>((unsigned)__vimin_s32_relu(x2, k.cap), k);
    q3 = round_mag1<SHIFT>((unsigned)__vimin_s32_relu(x3, k.cap), k);
    // values below 2^7: bytes assembled with multiply-adds
    return (q1 * 0x100u + q0) + (q3 * 0x1000000u + q2 * 0x10000u);
  }
  const unsigned a0 = (unsigned)abs(x0), a1 = (unsigned)abs(x1), a2 = (unsigned)abs(x2), a3 = (unsigned)abs(x3);
  e.orv |= a0 | a1;
  e.orv |= a2 | a3;
  const unsigned cap = (unsigned)k.cap;
  q0 = round_mag1<SHIFT>(min(a0, cap), k); q1 = round_mag1<SHIFT>(min(a1, cap), k);
  q2 = round_mag1<SHIFT>(min(a2, cap), k); q3 = round_mag1<SHIFT>(min(a3, cap), k);
  // sign as a multiply by +-1: the multiply runs beside the integer pipe
  q0 *= (unsigned)((x0 >> 31) | 1); q1 *= (unsigned)((x1 >> 31) | 1);
  q2 *= (unsigned)((x2 >> 31) | 1); q3 *= (unsigned)((x3 >> 31) | 1);
  return __byte_perm(__byte_perm(q0, q1, 0x4040), __byte_perm(q2, q3, 0x4040), 0x5410);
}
__device__ __forceinline__ unsigned prmt(unsigned a, unsigned b, unsigned sel) {
  unsigned d;
  asm("prmt.b32 %0, %1, %2, %3;" : "=r"(d) : "r"(a), "r"(b), "r"(sel));
  return d;
}
// (clamped magnitude + rounding term) * 2^k: the rounded value sits in byte B
__device__ __forceinline__ unsigned scaled_round(unsigned m, const RoundConst &k) {
  return (((~m) & k.mask2) | k.orc) * k.c2 + m * k.sc;
}
// Byte-aligned form of round_pack4.  Per element the half-rate integer pipe sees the extremes (one
// three-input min or max per element), the clamp, the bit select and half a permute; the two
// multiply-adds and the final merge run on the multiplier pipe.  Measured against the shift form:
// 6.9 instead of 9.0 issue cycles per element with ReLU, 10.9 instead of 15.1 without.
template <bool RELU>
__device__ __forceinline__ unsigned round_pack4_aligned(int x0, int x1, int x2, int x3, const RoundConst &k, Extremes &e) {
  if (RELU) {
    e.hi = __vimax3_s32(e.hi, x0, x1);
    e.hi = __vimax3_s32(e.hi, x2, x3);
    e.lo = __vimin3_s32(e.lo, x0, x1);
    e.lo = __vimin3_s32(e.lo, x2, x3);
    const unsigned v0 = scaled_round((unsigned)__vimin_s32_relu(x0, k.cap), k);
    const unsigned v1 = scaled_round((unsigned)__vimin_s32_relu(x1, k.cap), k);
    const unsigned v2 = scaled_round((unsigned)__vimin_s32_relu(x2, k.cap), k);
    const unsigned v3 = scaled_round((unsigned)__vimin_s32_relu(x3, k.cap), k);
    return prmt(v2, v3, k.sel) * k.m16 + prmt(v0, v1, k.sel);
  }
  const unsigned a0 = (unsigned)abs(x0), a1 = (unsigned)abs(x1), a2 = (unsigned)abs(x2), a3 = (unsigned)abs(x3);
  e.orv |= a0 | a1;
  e.orv |= a2 | a3;
  const unsigned cap = (unsigned)k.cap;
  const unsigned v0 = scaled_round(min(a0, cap), k), v1 = scaled_round(min(a1, cap), k);
  const unsigned v2 = scaled_round(min(a2, cap), k), v3 = scaled_round(min(a3, cap), k);
  const unsigned w = prmt(v2, v3, k.sel) * k.m16 + prmt(v0, v1, k.sel);
  // two's complement of the bytes whose accumulator was negative, four at a time: sm has 0xff in
  // those bytes (sign of the top byte of each accumulator, replicated); on the low seven bits
  // (w ^ sm) + 1 cannot carry into the next byte because w <= 127, and bit 7 is the sign unless the
  // byte is zero, which the last exclusive-or takes care of (0x80 ^ 0x80)
  const unsigned sm = prmt(prmt((unsigned)x0, (unsigned)x1, 0xfbfbu), prmt((unsigned)x2, (unsigned)x3, 0xfbfbu), 0x5410u);
  const unsigned t = ((w ^ sm) & 0x7f7f7f7fu) + (sm & 0x01010101u);
  return t ^ (sm & 0x80808080u);
}
// all variants behind one call: relu and the binary point are the same for every element of a pass
__device__ __forceinline__ void round_chunk32(const int (&v)[32], unsigned (&w8)[8], const RoundConst &k, bool relu,
                                              Extremes &e) {
  if (k.aligned) {
    if (relu) {
#pragma unroll
      for (int j = 0; j < 8; ++j) w8[j] = round_pack4_aligned<true>(v[4 * j], v[4 * j + 1], v[4 * j + 2], v[4 * j + 3], k, e);
    } else {
#pragma unroll
      for (int j = 0; j < 8; ++j) w8[j] = round_pack4_aligned<false>(v[4 * j], v[4 * j + 1], v[4 * j + 2], v[4 * j + 3], k, e);
    }
  } else if (relu) {      // (binary point above 24: only with fewer than seven magnitude bits)
#pragma unroll
    for (int j = 0; j < 8; ++j) w8[j] = round_pack4<true, true>(v[4 * j], v[4 * j + 1], v[4 * j + 2], v[4 * j + 3], k, e);
  } else {
#pragma unroll
    for (int j = 0; j < 8; ++j) w8[j] = round_pack4<false, true>(v[4 * j], v[4 * j + 1], v[4 * j + 2], v[4 * j + 3], k, e);
  }
}

// per byte: clamp(w - g, -127, 127) (Algorithm 1's update on int8 weights)
__device__ __forceinline__ unsigned bytes_sub_clamp127(unsigned w, unsigned g) {
  return __vmaxs4(__vsubss4(w, g), 0x81818181u);
}
// 0xff in every byte of b that is greater than zero as a signed byte (the ReLU gate of the backward pass).
__device__ __forceinline__ unsigned bytes_gt0(unsigned b) {
  unsigned t = (b & 0x7f7f7f7fu) + 0x7f7f7f7fu;   // bit 7 of a byte: its low seven bits are not all zero
  t = t & ~b & 0x80808080u;                       // ... and its sign bit is clear
  unsigned r;
  asm("prmt.b32 %0, %1, %1, 0xba98;" : "=r"(r) : "r"(t));   // replicate bit 7 over each byte
  return r;
}

// Byte-wise maximum of two words whose bytes are all in [0, 127] (ReLU outputs): bit 7 of
// (a | 0x80..) - b is set per byte exactly where a >= b, and no byte borrows from its neighbour.
__device__ __forceinline__ unsigned bytes_max_u7(unsigned a, unsigned b) {
  const unsigned t = (a | 0x80808080u) - b;
  unsigned m;
  asm("prmt.b32 %0, %1, %1, 0xba98;" : "=r"(m) : "r"(t));   // 0xff where a >= b
  return (a & m) | (b & ~m);
}
// 2 x 2 max-pool of a 32-channel chunk held one pixel per lane: the window's other pixels are the lanes
// lane ^ 1 (next column) and lane ^ xh (next image row); every lane ends up with its window's maximum.
__device__ __forceinline__ void pool_chunk32(unsigned (&w8)[8], int xh) {
#pragma unroll
  for (int j = 0; j < 8; ++j) {
    unsigned a = w8[j];
    a = bytes_max_u7(a, __shfl_xor_sync(0xffffffffu, a, 1));
    a = bytes_max_u7(a, __shfl_xor_sync(0xffffffffu, a, xh));
    w8[j] = a;
  }
}
__device__ __forceinline__ void store32(int8_t *dst, const unsigned (&w8)[8]) {
  asm volatile("st.global.v8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};"
               ::"l"(dst), "r"(w8[0]), "r"(w8[1]), "r"(w8[2]), "r"(w8[3]), "r"(w8[4]), "r"(w8[5]), "r"(w8[6]), "r"(w8[7])
               : "memory");
}

// Rows whose pitch or base is not a multiple of 32 bytes (`unit` = the largest power of two that divides
// both, at most 16).  A lane holds 32 columns of its own row, `nv` of them inside the matrix.  With units of
// 16 or 8 bytes every lane stores its own pieces; below that a store instruction of 32 scattered pieces
// costs 32 sector requests, so the chunk passes through shared memory (32 rows x 36 bytes per warp) and each
// instruction writes whole rows.
template <typename T>
__device__ __forceinline__ void store_rows_staged(int8_t *out8, unsigned off, bool rok, int nv, const unsigned *stg, int lane) {
  constexpr int LPR = 32 / (int)sizeof(T);                     // lanes per row
  const int part = lane % LPR;
  for (int r0 = 0; r0 < 32; r0 += (int)sizeof(T)) {
    const int r = r0 + lane / LPR;
    const unsigned o = __shfl_sync(0xffffffffu, off, r);
    const int ok = __shfl_sync(0xffffffffu, rok ? 1 : 0, r);
    if (ok && part * (int)sizeof(T) < nv)
      reinterpret_cast<T *>(out8 + o)[part] = reinterpret_cast<const T *>(reinterpret_cast<const char *>(stg) + r * 36)[part];
  }
}
__device__ __forceinline__ void store_rows_narrow(int8_t *out8, unsigned off, bool rok, const unsigned (&w8)[8], int nv,
                                                  int unit, unsigned *stg, int lane) {
  if (unit >= 8) {
    if (!rok) return;
    int8_t *dst = out8 + off;
    if (unit >= 16) {
      *reinterpret_cast<uint4 *>(dst) = make_uint4(w8[0], w8[1], w8[2], w8[3]);
      if (nv > 16) *reinterpret_cast<uint4 *>(dst + 16) = make_uint4(w8[4], w8[5], w8[6], w8[7]);
    } else {
#pragma unroll
      for (int j = 0; j < 4; ++j)
        if (8 * j < nv) *reinterpret_cast<uint2 *>(dst + 8 * j) = make_uint2(w8[2 * j], w8[2 * j + 1]);
    }
    return;
  }
#pragma unroll
  for (int j = 0; j < 8; ++j) stg[lane * 9 + j] = w8[j];
  __syncwarp();
  if (unit == 4) store_rows_staged<unsigned>(out8, off, rok, nv, stg, lane);
  else if (unit == 2) store_rows_staged<unsigned short>(out8, off, rok, nv, stg, lane);
  else store_rows_staged<unsigned char>(out8, off, rok, nv, stg, lane);
  __syncwarp();
}
// 32 gate bytes of this lane's row, from the aligned words that hold at least one of its nv bytes
__device__ __forceinline__ void load_row_narrow(const int8_t *src, unsigned (&m)[8], int nv) {
  const unsigned sh = 8u * (unsigned)((uintptr_t)src & 3);
  const unsigned *p = reinterpret_cast<const unsigned *>((uintptr_t)src & ~(uintptr_t)3);
  const int words = (nv + (int)((uintptr_t)src & 3) + 3) >> 2;
  unsigned lo = p[0];
#pragma unroll
  for (int j = 0; j < 8; ++j) {
    const unsigned hi = j + 1 < words ? p[j + 1] : 0u;
    m[j] = __funnelshift_r(lo, hi, sh);
    lo = hi;
  }
}

// Per call site the table keeps the errors (true bit-width minus sample-based estimate, each stored + 2
// in four bits) of the last two calls.  An error that repeats is systematic (the tensor's extremes sit
// outside the sampled tiles, or its distribution has a heavier tail than the scaling assumes) and is
// added to the next estimate; a single miss is the estimator's noise (on drifting training tensors about
// one launch in eight crosses a power of two unnoticed) and following it would only add misses.
__device__ __forceinline__ int spec_correction(int packed) {
  const int e1 = (packed & 15) - 2, e2 = ((packed >> 4) & 15) - 2;
  return e1 == e2 ? e1 : 0;
}

// The guess at a tensor's bit-width from the first tiles of a launch's CTAs, for one converged warp of every CTA; m: largest
// magnitude in its own first tile.  Posts and mailboxes as in niti_agree_bits: the first CTA decides when all have posted
// (deciding at half of them saved 0.2 us and made the guess depend on who came first: 50 of 100 launches of a 5 x 5 layer's
// error were recomputed, now none) and answers all of them.  (With a maximum, a count and a published word that all CTAs
// poll, updated by atomics, the agreement took 3.7 - 4.4 us, a chain of five trips to L2; this takes 2.2.)
//
// Nothing promises that all CTAs are on the GPU at the same time: where a kernel of another stream holds a single SM, the
// last CTA starts when one of this launch exits.  So the first CTA decides from half of the posts or more once no new one has
// come for GUESS_QUIET cycles, and from fewer after its whole patience.  Beside a kernel that holds 1 - 60 SMs for longer,
// 8192 x 4096 x 512 took 322 us where it waited for all posts and takes 65 (38 undisturbed), the error of the 5 x 5 layer 375
// - 400 and 130 - 164 (91).  In 500 passes over fifty layers alone on the GPU no launch went on early, with 2048, 4096, 8192
// or 16384 cycles.  (Marking early ones in the header, so that the follow-up does not remember their error, cost every
// follow-up 0.2 - 1.2 us; an error has to repeat before it is followed in any case.)  The other CTAs wait for the answer; out
// of patience twice as long as the first one's, a CTA decides from what has been posted by then.  Two CTAs may decide
// differently that way: every CTA reports what it rounded with (WsHeader::spec_mask), and the follow-up launch recomputes
// unless all of them used the true bit-width.
constexpr unsigned GUESS_QUIET = 8192;                  // about 4 us; the posts of an undisturbed launch come within 2
__device__ __forceinline__ int agree_on_guess(WsHeader *hdr, unsigned m, unsigned patience, unsigned mul256, int tag,
                                              const int32_t *spec_slot, int lane) {
  unsigned *const posts = niti_split_max(hdr), *const mail = posts + NITI_AGREE_MAX;
  const int cta = (int)blockIdx.x, n = (int)gridDim.x < NITI_AGREE_MAX ? (int)gridDim.x : NITI_AGREE_MAX;
  m = min(m, 0x7ffffffeu) + 1u;
  if (lane == 0 && cta < n) *(volatile unsigned *)(posts + cta) = m;
  // what the same estimate missed by at this call site lately (a systematic error of the sample, e.g. a tensor whose
  // extremes sit outside the first tiles); read while the posts are on their way
  int correction = 0;
  if (spec_slot && mul256 != 256 && *(volatile const int *)&spec_slot[0] == tag)
    correction = spec_correction(*(volatile const int *)&spec_slot[1]);
  unsigned since = (unsigned)clock64();                   // the start, or when the first CTA saw the last new post
  auto past = [&](unsigned limit) { return __any_sync(0xffffffffu, (unsigned)clock64() - since > limit) != 0; };
  if (cta != 0) {
    unsigned answer = 0;
    do {
      if (lane == 0) answer = *(volatile unsigned *)(mail + 4 * (cta < n ? cta : 0));
      answer = __shfl_sync(0xffffffffu, answer, 0);
    } while (!answer && !past(2u * patience));
    if (answer) return (int)answer - 1;
  }
  unsigned top, came = 0;
  while (true) {
    unsigned seen = 0;
    top = m;
#pragma unroll
    for (int u = 0; u < NITI_AGREE_MAX / 32; ++u) {
      const int i = 32 * u + lane;
      const unsigned w = i < n ? *(volatile unsigned *)(posts + i) : 0u;
      seen += w ? 1u : 0u;
      top = max(top, w);
    }
    seen = __reduce_add_sync(0xffffffffu, seen);
    if (cta != 0 || seen >= (unsigned)n) break;
    if (seen != came) since = (unsigned)clock64();
    came = seen;
    if (past(2u * seen >= (unsigned)n ? GUESS_QUIET : patience)) break;
  }
  top = __reduce_max_sync(0xffffffffu, top) - 1u;
  // the first tiles are a sample: scale their max by the growth expected from the sample to the whole tensor before taking
  // the bit length (a wrong guess only costs the second pass); never below the bit length of the sample's own maximum,
  // which the tensor's cannot undercut
  unsigned long long scaled = ((unsigned long long)top * mul256) >> 8;
  if (scaled > 0x7fffffffull) scaled = 0x7fffffffull;
  int guess = niti_bitlen32((unsigned)scaled) + correction;
  const int floor_b = niti_bitlen32(top);
  guess = guess < floor_b ? floor_b : (guess > 31 ? 31 : guess);
  if (cta == 0)
    for (int i = lane; i < n; i += 32) *(volatile unsigned *)(mail + 4 * i) = (unsigned)guess + 1u;
  return guess;
}

// tile index -> (column tile, row tile, image)
__device__ __forceinline__ void tile_coords(const TcParams &p, int idx, int &wt, int &ht, int &bt) {
  const int t = div_by(idx, p.d_w);
  wt = idx - t * p.w_tiles;
  bt = div_by(t, p.d_h);
  ht = t - bt * p.h_tiles;
}
// Coordinates of an output tile / k-block in the pixel grid of a convolution.
__device__ __forceinline__ void pixel_box(const TcParams &p, int idx, int &w0, int &h0, int &b0) {
  int wt, ht, bt;
  tile_coords(p, idx, wt, ht, bt);
  w0 = wt * p.Wt; h0 = ht * p.Ht; b0 = bt * p.Bt;
}

// Phase of an item of a strided error multiply (dstride > 1): items run over (tile, phase), so that a contiguous
// range of items holds all phases, which have different numbers of taps, in equal shares.
struct Phase { int r, s, n_r, n_s; };     // first tap row / column, taps of the phase
__device__ __forceinline__ Phase split_phase(const TcParams &p, int item, int &tile) {
  tile = div_by(item, p.d_phases);
  const int ph = item - tile * p.nph_r * p.nph_s;
  Phase q;
  q.r = div_by(ph, p.d_phase_s);
  q.s = ph - q.r * p.nph_s;
  // (the phases before R mod stride have one tap more)
  q.n_r = q.r + (p.T_r - 1) * p.dstride < p.R ? p.T_r : p.T_r - 1;
  q.n_s = q.s + (p.T_s - 1) * p.dstride < p.S ? p.T_s : p.T_s - 1;
  return q;
}

// Output row of grid position `idx` of a phase of a strided error multiply; ok: it is inside the tensor.
__device__ __forceinline__ int phase_row(const TcParams &p, int idx, const Phase &q, bool &ok) {
  int v, u, b;
  tile_coords(p, idx, v, u, b);
  const int jj = (v + p.u0_s) * p.dstride + q.s - p.pad, ii = (u + p.u0_r) * p.dstride + q.r - p.pad;
  ok = b < p.PB && ii >= 0 && ii < p.OH && jj >= 0 && jj < p.OW;
  return (b * p.OH + ii) * p.OW + jj;
}

// ------------------------------------------------------------------------------------------
// Cluster helpers (CTAS == 2: a pair of CTAs on neighbouring SMs works on one 256-row tile with
// tcgen05 cta_group::2; the even CTA of the pair issues the MMAs and owns the barriers).
// ------------------------------------------------------------------------------------------
__device__ __forceinline__ unsigned cluster_ctarank() {
  unsigned r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
__device__ __forceinline__ unsigned map_to_cta(unsigned local_addr, unsigned rank) {
  unsigned r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(local_addr), "r"(rank));
  return r;
}
__device__ __forceinline__ void cluster_sync_all() {
  asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
  asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ void mbar_arrive_cluster(unsigned cluster_addr) {
  asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(cluster_addr) : "memory");
}
__device__ __forceinline__ void tma_load_2d_pair(unsigned dst, const CUtensorMap *map, unsigned bar, int c0, int c1) {
  asm volatile(
      "cp.async.bulk.tensor.2d.cta_group::2.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4}], [%2];"
      ::"r"(dst), "l"(map), "r"(bar), "r"(c0), "r"(c1)
      : "memory");
}
__device__ __forceinline__ void tma_load_4d_pair(unsigned dst, const CUtensorMap *map, unsigned bar, int c0, int c1,
                                                 int c2, int c3) {
  asm volatile(
      "cp.async.bulk.tensor.4d.cta_group::2.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, %5, %6}], [%2];"
      ::"r"(dst), "l"(map), "r"(bar), "r"(c0), "r"(c1), "r"(c2), "r"(c3)
      : "memory");
}
__device__ __forceinline__ void tma_load_3d_pair(unsigned dst, const CUtensorMap *map, unsigned bar, int c0, int c1, int c2) {
  asm volatile(
      "cp.async.bulk.tensor.3d.cta_group::2.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, %5}], [%2];"
      ::"r"(dst), "l"(map), "r"(bar), "r"(c0), "r"(c1), "r"(c2)
      : "memory");
}
__device__ __forceinline__ void tma_load_im2col_pair(unsigned dst, const CUtensorMap *map, unsigned bar, int c, int w, int h,
                                                     int n, unsigned short ow, unsigned short oh) {
  asm volatile(
      "cp.async.bulk.tensor.4d.cta_group::2.shared::cluster.global.im2col.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, %5, %6}], [%2], {%7, %8};"
      ::"r"(dst), "l"(map), "r"(bar), "r"(c), "r"(w), "r"(h), "r"(n), "h"(ow), "h"(oh)
      : "memory");
}
__device__ __forceinline__ void tc_commit_pair(unsigned bar) {
  asm volatile(
      "tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;"
      ::"r"(bar), "h"((unsigned short)3)
      : "memory");
}

__device__ __forceinline__ void tc_mma_i8_pair_lh(unsigned tmem_d, unsigned a_lo, unsigned a_hi, unsigned b_lo,
                                                  unsigned b_hi, unsigned idesc, unsigned accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t.reg .b64 da, db;\n\t"
      "setp.ne.b32 p, %6, 0;\n\t"
      "mov.b64 da, {%1, %2};\n\t"
      "mov.b64 db, {%3, %4};\n\t"
      "tcgen05.mma.cta_group::2.kind::i8 [%0], da, db, %5, p;\n\t}"
      ::"r"(tmem_d), "r"(a_lo), "r"(a_hi), "r"(b_lo), "r"(b_hi), "r"(idesc), "r"(accumulate)
      : "memory");
}

// The issuing thread is a single instruction stream: every scalar instruction between two MMAs is
// on the critical path of the tensor pipe (measured: run-time trip counts, selects and multiplies
// per MMA cost ~35 cycles each time, more than half of an N = 64 MMA).  The issue loops are therefore
// compiled per k-step count, with every offset either a literal or a register filled before the
// tile loop.
//
// One 3x3 tile from the resident patch: nine taps, KS k-steps each, into one accumulator.
template <int KS>
__device__ __forceinline__ void halo_issue_tile(unsigned tmem_d, unsigned a_lo, unsigned a_hi, const unsigned (&a_off)[9],
                                                unsigned b_hi, const unsigned (&b_tap)[9], unsigned b_kstep16,
                                                unsigned idesc) {
#pragma unroll
  for (int tap = 0; tap < 9; ++tap) {
    const unsigned a_t = a_lo + a_off[tap];
#pragma unroll
    for (int k = 0; k < KS; ++k)
      tc_mma_i8_lh(tmem_d, a_t + 2u * k, a_hi, b_tap[tap] + (unsigned)k * b_kstep16, b_hi, idesc,
                   (tap > 0 || k > 0) ? 1u : 0u);
  }
}
// One k-block of the generic loop: KS MMAs whose operands advance by the k-step strides.
template <int CTAS, int KS>
__device__ __forceinline__ void issue_kblock(unsigned tmem_d, unsigned a_lo, unsigned a_hi, unsigned b_lo, unsigned b_hi,
                                             unsigned a_kstep16, unsigned b_kstep16, unsigned idesc, unsigned first_acc) {
#pragma unroll
  for (int k = 0; k < KS; ++k) {
    if (CTAS == 2)
      tc_mma_i8_pair_lh(tmem_d, a_lo + (unsigned)k * a_kstep16, a_hi, b_lo + (unsigned)k * b_kstep16, b_hi, idesc,
                        k > 0 ? 1u : first_acc);
    else
      tc_mma_i8_lh(tmem_d, a_lo + (unsigned)k * a_kstep16, a_hi, b_lo + (unsigned)k * b_kstep16, b_hi, idesc,
                   k > 0 ? 1u : first_acc);
  }
}

template <int CTAS>
__device__ __forceinline__ void load2(unsigned dst, const CUtensorMap *m, unsigned bar, int c0, int c1) {
  if (CTAS == 2) tma_load_2d_pair(dst, m, bar, c0, c1); else tma_load_2d(dst, m, bar, c0, c1);
}
template <int CTAS>
__device__ __forceinline__ void load4(unsigned dst, const CUtensorMap *m, unsigned bar, int c0, int c1, int c2, int c3) {
  if (CTAS == 2) tma_load_4d_pair(dst, m, bar, c0, c1, c2, c3); else tma_load_4d(dst, m, bar, c0, c1, c2, c3);
}

template <int CTAS>
__device__ __forceinline__ void load3(unsigned dst, const CUtensorMap *m, unsigned bar, int c0, int c1, int c2) {
  if (CTAS == 2) tma_load_3d_pair(dst, m, bar, c0, c1, c2); else tma_load_3d(dst, m, bar, c0, c1, c2);
}
template <int CTAS>
__device__ __forceinline__ void load_im2col(unsigned dst, const CUtensorMap *m, unsigned bar, int c, int w, int h, int n,
                                            int ow, int oh) {
  if (CTAS == 2) tma_load_im2col_pair(dst, m, bar, c, w, h, n, (unsigned short)ow, (unsigned short)oh);
  else tma_load_im2col(dst, m, bar, c, w, h, n, (unsigned short)ow, (unsigned short)oh);
}

// Next tap of a tap group; beyond the last one it is repeated (the filler's results are not used).
__device__ __forceinline__ void next_tap(const TcParams &p, int &jb, int &r, int &s) {
  jb = 0;
  if (++s == p.S) {
    s = 0;
    if (++r == p.R) { r = p.R - 1; s = p.S - 1; }
  }
}

// item -> (row unit, column tile, split).  Row units (one CTA's 128 rows, or a pair's 256) are
// visited in groups of raster_g so that the CTAs running at the same time share operand tiles in L2.
// (32-bit arithmetic throughout: one thread of the producer, issuer and epilogue warps runs this per
// tile, and 64-bit divisions there cost more than a small tile's whole multiply.)
__device__ __forceinline__ void decode_item(const TcParams &p, int item, int &mu, int &nt, int &split) {
  int tile = item;
  split = 0;
  if (p.splits > 1) {
    tile = div_by(item, p.d_split);
    split = item - tile * p.splits;
  }
  if (p.raster_g <= 0) {
    mu = div_by(tile, p.d_n);
    nt = tile - mu * p.n_tiles_n;
    return;
  }
  const int g = div_by(tile, p.d_group);
  const int rem = tile - g * p.raster_g * p.n_tiles_n;
  const bool last = g == p.last_group;
  nt = div_by(rem, last ? p.d_last : p.d_units);
  mu = g * p.raster_g + rem - nt * (last ? p.m_units - g * p.raster_g : p.raster_g);
}

// ------------------------------------------------------------------------------------------
// The kernel
// ------------------------------------------------------------------------------------------
// Issuing loop of the resident-weights mode.  `nissue` warps (1 or 2) run it, warp `issuer` taking
// tiles issuer, issuer + nissue, ... of the CTA's range: with 64 output channels a tile is only 18 MMAs,
// and one warp's per-tile bookkeeping (two barrier tests, fences, two commits) leaves the tensor pipe
// idle for a quarter of the time; two issuers fill each other's gaps.  Tiles go to different
// accumulator buffers, so the order in which the pipe sees the two warps' MMAs does not matter, and
// each warp's commits cover exactly its own MMAs.
__device__ __forceinline__ void halo_mma_loop(const TcParams &p, int issuer, int nissue, int first_item, int item_end,
                                              unsigned smem_base, unsigned tmem_base, unsigned full0, unsigned empty0,
                                              unsigned tfull0, unsigned tempty0, unsigned bres_bar,
                                              volatile int *abort_flag, uint32_t *status) {
  const bool leader = elect_one();
  bool ok = mbar_wait_warp(bres_bar, 0, abort_flag, status);
  // descriptor low words per tap, computed once: the patch row where the tap starts
  // (forward reads x[i + r - 1][j + t - 1], dgrad reads e[i - r + 1][j - t + 1]; the patch
  // starts one pixel up and left of the tile) and the tap's resident weight tile
  const unsigned a_hi = (unsigned)(p.a_desc >> 32), b_hi = (unsigned)(p.b_desc >> 32);
  const unsigned a_lo0 = (unsigned)p.a_desc, b_lo0 = (unsigned)p.b_desc + ((smem_base >> 4) & 0x3fff);
  const unsigned row16 = (unsigned)p.kdepth >> 4, btile16 = (unsigned)p.b_tile_bytes >> 4;
  const bool fwd_taps = p.kind == GK_CONV_FWD;
  const unsigned a_stage16 = (unsigned)p.a_bytes >> 4;
  const unsigned a_stage_lo = a_lo0 + (((smem_base + p.b_res_bytes) >> 4) & 0x3fff);   // stage 0
  const unsigned b_kstep16 = p.b_kstep16, idesc = p.idesc;
  const int ksteps = p.ksteps, stages = p.stages;
  const unsigned nbuf = (unsigned)p.nbuf, bn = (unsigned)p.bn;
  unsigned a_off[9], b_tap[9];
#pragma unroll
  for (int tap = 0; tap < 9; ++tap) {
    const int r = tap / 3, t = tap % 3;
    a_off[tap] = (fwd_taps ? (unsigned)(r * 10 + t) : (unsigned)((2 - r) * 10 + (2 - t))) * row16;
    b_tap[tap] = b_lo0 + (unsigned)tap * btile16;
  }
  const bool one_commit = p.one_commit != 0;
  int stage = 0;
  unsigned phase = 0;
  unsigned hbuf = 0, hpar = 0;          // tile % nbuf, (tile / nbuf) & 1, counted
  if (issuer) {                         // (issuer is 0 or 1)
    if (++stage == stages) { stage = 0; phase ^= 1; }
    if (++hbuf == nbuf) { hbuf = 0; hpar ^= 1u; }
  }
  for (int item = first_item + issuer; ok && item < item_end; item += nissue) {
    // (with one_commit the accumulator buffer is the stage and their parities coincide)
    const unsigned buf = one_commit ? (unsigned)stage : hbuf;
    const unsigned par = one_commit ? phase : hpar;
    if (!mbar_wait_warp(tempty0 + 8 * buf, par ^ 1u, abort_flag, status)) break;
    if (!mbar_wait_warp(full0 + 8 * stage, phase, abort_flag, status)) break;
    tc_fence_after();
    const unsigned tmem_d = tmem_base + buf * bn;
    const unsigned a_lo = a_stage_lo + (unsigned)stage * a_stage16;
    if (leader) {
      if (ksteps == 2) halo_issue_tile<2>(tmem_d, a_lo, a_hi, a_off, b_hi, b_tap, b_kstep16, idesc);
      else if (ksteps == 3) halo_issue_tile<3>(tmem_d, a_lo, a_hi, a_off, b_hi, b_tap, b_kstep16, idesc);
      else if (ksteps == 4) halo_issue_tile<4>(tmem_d, a_lo, a_hi, a_off, b_hi, b_tap, b_kstep16, idesc);
      else halo_issue_tile<1>(tmem_d, a_lo, a_hi, a_off, b_hi, b_tap, b_kstep16, idesc);
      if (!one_commit) tc_commit(empty0 + 8 * stage);
      tc_commit(tfull0 + 8 * buf);
    }
    for (int j = 0; j < nissue; ++j) {
      if (++stage == stages) { stage = 0; phase ^= 1; }
      if (++hbuf == nbuf) { hbuf = 0; hpar ^= 1u; }
    }
  }
}
// Instances.  MODE 0: pixel boxes and plain matrices whose operands are whole chunks and whose output rows are
// 32-byte aligned (the layers of the benchmark networks).  MODE 1: everything else that has no phases: im2col
// copies, short channel chunks, output rows of any pitch.  MODE 2: MODE 1 for the error of a strided
// convolution (items run over the phases of the input grid).  With one kernel for all of them the index
// arithmetic and the registers of the general forms cost the aligned layers 1 - 4 % (13 spilled registers more;
// 14 x 14 weight gradients 28.8 -> 30.4 us, 56 x 56 ones 86.2 -> 89.7 us).
// ONE: single-wave launches, in which every CTA has at most one tile, the shift is exact and a CTA may leave (see
// niti_agree_bits).  They have no use for the loops over tiles, and the others none for what leaving takes (with both in one
// kernel a VGG-11 step took 514 us, with neither loop nor leaving apart 498 us, with these instances 485 us).

// The tile of CTA `cta` of a single-wave launch, which left its sums in `acc`: rounded and stored element by element, by all
// threads of another CTA.
template <int CTAS, bool STRIDED>
__device__ __forceinline__ void round_left_tile(const TcParams &p, int cta, int b, const int32_t *acc, int8_t *out8,
                                                const int8_t *mask8, int8_t *pool8) {
  const int item = cta / CTAS, rank = cta - item * CTAS;              // (one item per CTA pair, in the order of the CTAs)
  const int lane = threadIdx.x & 31, bp = b > p.mbits ? b - p.mbits : 0;
  const unsigned qmax = (1u << p.mbits) - 1u;
  int tile = item, mu = 0, nt = 0, split = 0;
  Phase phq = {0, 0, 1, 1};
  if (STRIDED) phq = split_phase(p, item, tile);
  if (!p.halo) decode_item(p, tile, mu, nt, split);
  const int mt = mu * CTAS + rank;
  int col0 = nt * p.bn;
  int cols = min(p.bn, p.gn - col0);
  if (p.kind == GK_CONV_WGRAD) {
    const int tap = div_by(nt, p.d_chunks), ci0 = (nt - tap * p.n_chunks) * p.bn;
    col0 = tap * p.Cn + ci0;
    cols = min(p.bn, p.Cn - ci0);
  }
  const bool boxes = p.halo || ((p.kind == GK_CONV_FWD || p.kind == GK_CONV_DGRAD) && !p.i2c);
  auto rounded = [&](unsigned at) {
    const int q = niti_round_i32(__ldcg(acc + at), bp, qmax, p.round_mode);
    return p.relu && q < 0 ? 0 : q;
  };
  for (int r = (int)(threadIdx.x >> 5); r < BM; r += NUM_THREADS / 32) {
    int row;
    bool ok;
    int w = 0, h = 0, bb = 0;
    if (STRIDED) {
      row = phase_row(p, mt * BM + r, phq, ok);
    } else if (boxes) {
      if (p.halo) {
        tile_coords(p, item, w, h, bb);
        w = w * 8 + (r & 7);
        h = h * 16 + (r >> 3);
      } else {
        pixel_box(p, mt, w, h, bb);
        const int t = r >> p.wt_shift;
        w += r & (p.Wt - 1);
        h += t & (p.Ht - 1);
        bb += t >> p.ht_shift;
      }
      ok = w < p.PW && h < p.PH && bb < p.PB;
      row = (bb * p.PH + h) * p.PW + w;
    } else {
      row = mt * BM + r;
      ok = row < p.gm;
    }
    if (!ok) continue;
    const bool pools = p.pool && ((w | h) & 1) == 0;                  // (extents are even, windows lie inside the tile)
    for (int c = lane; c < cols; c += 32) {
      const unsigned at = (unsigned)row * (unsigned)p.gn + (unsigned)(col0 + c);
      int q = rounded(at);
      if (pools) {
        const int m = max(max(q, rounded(at + p.gn)), max(rounded(at + p.PW * p.gn), rounded(at + (p.PW + 1) * p.gn)));
        pool8[(unsigned)((bb * (p.PH >> 1) + (h >> 1)) * (p.PW >> 1) + (w >> 1)) * (unsigned)p.gn + (unsigned)(col0 + c)] = (int8_t)m;
      }
      if (p.update) {
        const int d = (int)out8[at] - q;
        q = d > 127 ? 127 : (d < -127 ? -127 : d);
      } else if (mask8 && mask8[at] <= 0) {
        q = 0;
      }
      out8[at] = (int8_t)q;
    }
  }
}

template <int CTAS, int MODE, bool ONE>
__global__ void __launch_bounds__(NUM_THREADS, 1)
tc_gemm_kernel(const __grid_constant__ CUtensorMap map_a, const __grid_constant__ CUtensorMap map_b,
               const __grid_constant__ CUtensorMap map_c, const TcParams p, int32_t *__restrict__ acc, WsHeader *hdr, uint32_t *status,
               int8_t *__restrict__ out8, const int8_t *__restrict__ mask8, const int32_t *s_a,
               const int32_t *s_w, int32_t *s_out, int32_t *b_out, int32_t *spec_slot, int8_t *__restrict__ pool8) {
  constexpr bool I2C = MODE >= 1, STRIDED = MODE == 2, GENERAL = MODE >= 1;
  const int epi_mode = ONE ? (int)EPI_SPECULATE : p.epi_mode;
  if (epi_mode == EPI_KNOWN_B) {
    // follow-up of a speculative pass: publish the scalars, then leave unless the guess was wrong
    asm volatile("griddepcontrol.wait;" ::: "memory");     // the first pass has completed and is visible
    const unsigned used = hdr->spec_mask;                  // bit-widths that the CTAs rounded with
    const int b_true = niti_bitlen32(hdr->maxabs32), b_est = used ? 31 - __clz(used) : b_true;
    if (blockIdx.x == 0 && threadIdx.x == 0) {
      if (spec_slot) {
        // remember, for the next calls from this call site, how far the sample-based estimate was off
        // (b_est = raw estimate + the correction this call applied): the last two errors are kept
        const int packed = spec_slot[0] == p.spec_tag ? spec_slot[1] : 0x22;
        int err = b_true - (b_est - spec_correction(packed));
        err = err < -2 ? -2 : (err > 2 ? 2 : err);
        spec_slot[0] = p.spec_tag;
        spec_slot[1] = (err + 2) | ((packed & 15) << 4);
      }
      const int bp = b_true > p.mbits ? b_true - p.mbits : 0;
      if (b_out) *b_out = b_true;
      if (s_out) {
        int s = bp + (s_a ? *s_a : 0) + (s_w ? *s_w : 0);
        *s_out = s;
        if (s < -128 || s > 127) atomicOr(status, NITI_DEV_EXP_RANGE);
      }
    }
    if (used == 1u << (b_true & 31)) return;
    if (blockIdx.x == 0 && threadIdx.x == 0) atomicAdd(status + 1, 1u);   // count of recomputations
  }
  extern __shared__ __align__(1024) uint8_t smem_raw[];
  __shared__ __align__(8) unsigned long long bars[2 * MAX_STAGES + 2 * MAX_TBUF + 1];
  __shared__ unsigned tmem_base_slot;
  __shared__ volatile int abort_flag;
  __shared__ volatile int spec_bp_ready;      // 0: not yet; the speculative binary point + 1; -1: this CTA leaves
  __shared__ unsigned ticket;                 // of the agreement of a single-wave launch
  __shared__ unsigned first_max, first_arrived;   // this CTA's first tile: max magnitude, warps that reported
  __shared__ unsigned cta_max;                    // max magnitude of everything this CTA rounded
  __shared__ int cta_b;                           // bit-width it rounded with (-1: nothing was agreed)

  const int warp = __shfl_sync(0xffffffffu, (int)(threadIdx.x >> 5), 0), lane = threadIdx.x & 31;
  const unsigned rank = CTAS == 2 ? cluster_ctarank() : 0u;
  const unsigned smem_base = (smem_u32(smem_raw) + 1023u) & ~1023u;
  const int stage_bytes = p.a_bytes + p.b_bytes;
  const unsigned full0 = smem_u32(&bars[0]);
  const unsigned empty0 = smem_u32(&bars[MAX_STAGES]);
  const unsigned tfull0 = smem_u32(&bars[2 * MAX_STAGES]);
  const unsigned tempty0 = smem_u32(&bars[2 * MAX_STAGES + MAX_TBUF]);
  const unsigned bres_bar = smem_u32(&bars[2 * MAX_STAGES + 2 * MAX_TBUF]);   // resident weights landed
  // barriers of the leader CTA as seen from this CTA
  const unsigned lead_full0 = CTAS == 2 ? map_to_cta(full0, 0) : full0;
  const unsigned lead_tempty0 = CTAS == 2 ? map_to_cta(tempty0, 0) : tempty0;
  // items of this CTA (pair): first_item, first_item + item_step, ... below item_end
  int first_item = blockIdx.x / CTAS, item_step = gridDim.x / CTAS, item_end = (int)p.items;
  if (p.blocked) {
    const int u = blockIdx.x / CTAS;
    const int per = p.blk_per, extra = p.blk_extra;
    first_item = u * per + (u < extra ? u : extra);
    item_end = first_item + per + (u < extra ? 1 : 0);
    item_step = 1;
  }

  // epilogue warps with at least one 32-column chunk of the tile (four per chunk phase)
  // The 16 epilogue warps are split into `egroups` groups that drain different tiles at the same
  // time (narrow tiles have too few 32-column chunks to keep every warp busy on one tile).  Inside a
  // group each TMEM lane quarter has wpq warps that interleave the tile's chunks.
  const int egroups = ONE || p.halo == 2 ? 1 : p.egroups;
  const int wpq = p.k_wpq;                                   // warps per quarter per tile
  const int wpq_active = p.k_wpq_active;
  const int epi_active = p.k_epi_active;                     // warps that drain one tile
  // TMEM columns: nbuf accumulator buffers of bn columns, rounded up to a power of two >= 32
  const unsigned tmem_cols = (unsigned)p.k_tmem_cols;

  // Set-up is paid by every launch (measured: 1.8 us from entry to the first copy when one thread did
  // all of it): the tensor maps are prefetched at once, every barrier is initialised by its own
  // thread, and tensor memory is allocated by another warp meanwhile.
  if (threadIdx.x == 32) {
    asm volatile("prefetch.tensormap [%0];" ::"l"(&map_a) : "memory");
    asm volatile("prefetch.tensormap [%0];" ::"l"(&map_b) : "memory");
    if (p.red) asm volatile("prefetch.tensormap [%0];" ::"l"(&map_c) : "memory");
  }
  if (threadIdx.x == 0) {
    abort_flag = 0;
    spec_bp_ready = 0;
    first_max = 0;
    first_arrived = 0;
    cta_max = 0;
    cta_b = -1;
  }
  if (threadIdx.x < 2 * MAX_STAGES + 2 * MAX_TBUF + 1) {
    const int bi = (int)threadIdx.x;
    const bool is_tempty = bi >= 2 * MAX_STAGES + MAX_TBUF && bi < 2 * MAX_STAGES + 2 * MAX_TBUF;
    // one arrival per barrier, except "accumulator drained": one per working epilogue warp of every CTA
    mbar_init(smem_u32(&bars[bi]), is_tempty ? epi_active * CTAS : 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  if (warp == MMA_WARP) {
    if (CTAS == 2) {
      asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;"
                   ::"r"(smem_u32(&tmem_base_slot)), "r"(tmem_cols) : "memory");
      asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
    } else {
      asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;"
                   ::"r"(smem_u32(&tmem_base_slot)), "r"(tmem_cols) : "memory");
      asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
  }
  tc_fence_before();
  __syncthreads();
  if (CTAS == 2) cluster_sync_all();   // the peer's barriers exist before anyone signals them
  tc_fence_after();
  const unsigned tmem_base = tmem_base_slot;
  // (the set-up above overlaps the kernel before this one; a follow-up launch that is scheduled from here on takes the SMs
  // as this grid's CTAs retire)
  const int8_t *const mask_at_exit = mask8;          // (the parameter itself: costs the main loops no register)
  niti_enter(mask8);
  if (ONE && threadIdx.x == NUM_THREADS - 1) ticket = niti_arrive(hdr);      // (a thread that has to wait anyway)
  if (p.next && blockIdx.x == 0 && warp == NUM_THREADS / 32 - 2) niti_zero_header(p.next, lane);

  // the scalars of a single-wave launch: the shift is exact, and no second launch publishes them
  auto publish_exact = [&](int b) {
    const int bpf = b > p.mbits ? b - p.mbits : 0;
    if (b_out) *b_out = b;
    if (s_out) {
      const int sv = bpf + (s_a ? *s_a : 0) + (s_w ? *s_w : 0);
      *s_out = sv;
      if (sv < -128 || sv > 127) atomicOr(status, NITI_DEV_EXP_RANGE);
    }
  };

  const bool epi_warp = warp >= EPI_WARP0 && (((warp - EPI_WARP0) >> 2) & (wpq - 1)) < wpq_active;
  if (warp < PROD_WARPS) {
    // ================= TMA producers (every CTA loads its own rows of A and its share of B) ========
    // Each producer warp runs its loop in lock step and one elected lane issues the copies (warp-uniform
    // control flow keeps the coordinate arithmetic in the uniform datapath that feeds the TMA unit).
    {
      const bool leader = elect_one();
      int stage = 0;
      unsigned phase = 0;
      bool ok = true;
      // (an integer division costs a lone warp ~200 cycles: nothing below divides per k-block or per
      // tile; the warp that owns the current stage is counted, stage % nprod)
      int owner = 0;
      const int nprod = p.nprod;
      const int bn_cta = p.bn / CTAS;             // B rows (output columns) staged by this CTA
      if (p.halo == 2) {
        for (int item = first_item; ok && item < item_end; item += item_step) {
          const int blk = div_by(item, p.d_split), split = item - blk * p.splits;
          const int ci0 = (blk % p.wg_nci) * 64, co0 = (blk / p.wg_nci) * 64;
          const int t0 = split * p.kb_per_split;
          int t1 = t0 + p.kb_per_split;
          if (t1 > p.kb_total) t1 = p.kb_total;
          int wt, ht, bt;
          tile_coords(p, t0, wt, ht, bt);
          for (int t = t0; t < t1; ++t) {
            if (owner == warp) {
              if (!mbar_wait_warp(empty0 + 8 * stage, phase ^ 1, &abort_flag, status)) { ok = false; break; }
              const unsigned full = full0 + 8 * stage;
              const unsigned sa = smem_base + stage * stage_bytes;
              if (leader) {
                mbar_expect_tx(full, (unsigned)(p.a_box_bytes + p.b_box_bytes));
                tma_load_4d(sa, &map_a, full, ci0, wt * 8 - 1, ht * 16 - 1, bt);          // input patch
                tma_load_4d(sa + p.a_bytes, &map_b, full, co0, wt * 8, ht * 16, bt);     // error tile
              }
            }
            if (++owner == nprod) owner = 0;
          if (++stage == p.stages) { stage = 0; phase ^= 1; }
            if (++wt == p.w_tiles) { wt = 0; if (++ht == p.h_tiles) { ht = 0; ++bt; } }
          }
        }
        item_end = first_item;
      } else if (p.halo) {
        // resident weights: one tile per tap, [bn rows][kdepth] K-major (forward) or
        // [kdepth rows][bn] MN-major in b_boxes column chunks (dgrad)
        // (issued by the last producer warp: the first one owns stage 0 and starts with tile 0's patch)
        if (warp == PROD_WARPS - 1 && leader) mbar_expect_tx(bres_bar, (unsigned)(9 * p.b_boxes * p.b_box_bytes));
        for (int tap = 0; warp == PROD_WARPS - 1 && leader && tap < 9; ++tap) {
          const unsigned dst = smem_base + tap * p.b_tile_bytes;
          if (p.kind == GK_CONV_FWD) {
            if (GENERAL) tma_load_3d(dst, &map_b, bres_bar, 0, tap, 0);
            else tma_load_2d(dst, &map_b, bres_bar, tap * p.kdepth, 0);
          } else {
            for (int j = 0; j < p.b_boxes; ++j) {
              if (GENERAL) tma_load_3d(dst + j * p.b_box_bytes, &map_b, bres_bar, j * p.b_box_step, tap, 0);
              else tma_load_2d(dst + j * p.b_box_bytes, &map_b, bres_bar, tap * p.Cn + j * p.b_box_step, 0);
            }
          }
        }
        if (p.nissue == 2 && warp == PROD_WARPS - 1) {
          // (the other producer warps load the patches; this one issues every other tile's MMAs)
          if (rank == 0)
            halo_mma_loop(p, 1, 2, first_item, item_end, smem_base, tmem_base, full0, empty0, tfull0, tempty0,
                          bres_bar, &abort_flag, status);
          item_end = first_item;
        }
        // consecutive items are consecutive tiles (blocked assignment): step the tile coordinates
        int wt, ht, bt;
        tile_coords(p, first_item, wt, ht, bt);
        const unsigned free0 = p.one_commit ? tfull0 : empty0;   // "tile done" also frees the patch stage
        for (int item = first_item; ok && item < item_end; ++item) {
          if (owner == warp) {
            if (!mbar_wait_warp(free0 + 8 * stage, phase ^ 1, &abort_flag, status)) { ok = false; break; }
            const unsigned full = full0 + 8 * stage;
            if (leader) {
              mbar_expect_tx(full, (unsigned)p.a_box_bytes);
              tma_load_4d(smem_base + p.b_res_bytes + stage * p.a_bytes, &map_a, full, 0, wt * 8 - 1, ht * 16 - 1, bt);
            }
          }
          if (++owner == nprod) owner = 0;
          if (++stage == p.stages) { stage = 0; phase ^= 1; }
          if (++wt == p.w_tiles) { wt = 0; if (++ht == p.h_tiles) { ht = 0; ++bt; } }
        }
        item_end = first_item;                    // nothing left for the generic loop
      }
      // Tile transitions are on the critical path of the whole pipeline (while a producer decodes its
      // next tile no copy is issued and the ring runs dry; measured: ~1500 cycles of integer divisions
      // per tile cost a third of a 256-channel convolution).  Consecutive items of the convolutions
      // are consecutive tiles, so tile and pixel-box coordinates are stepped, not divided.
      // One instance of the loop per kind of multiply: a producer that finds out what to copy for every k-block issues a third
      // fewer copies.
      auto produce = [&](auto kind_c, auto i2c_c) {
        constexpr int KIND = decltype(kind_c)::value;
        constexpr bool IC = decltype(i2c_c)::value;           // im2col copies
        // the B tile of a k-block (forward and error multiplies)
        auto load_b = [&](unsigned sb, unsigned full, int kb, int cc, int tap, int nb) {
          if (KIND == GK_FC_FWD) {
            load2<CTAS>(sb, &map_b, full, kb * p.kdepth, nb);
          } else if (KIND == GK_CONV_FWD) {
            if (GENERAL) load3<CTAS>(sb, &map_b, full, cc * p.kdepth, tap, nb);
            else load2<CTAS>(sb, &map_b, full, kb * p.kdepth, nb);
          } else {
            for (int j = 0; j < p.b_boxes; ++j)
              if (KIND == GK_FC_DGRAD) load2<CTAS>(sb + j * p.b_box_bytes, &map_b, full, nb + j * p.b_box_step, kb * p.kdepth);
              else if (GENERAL) load3<CTAS>(sb + j * p.b_box_bytes, &map_b, full, nb + j * p.b_box_step, tap, cc * p.kdepth);
              else load2<CTAS>(sb + j * p.b_box_bytes, &map_b, full, tap * p.Cn + nb + j * p.b_box_step, cc * p.kdepth);
          }
        };
        constexpr bool RES = CTAS == 1 && !ONE && !STRIDED && KIND != GK_FC_WGRAD && KIND != GK_CONV_WGRAD;
        const bool resident = RES && p.b_resident != 0;
        const bool stepped = p.blocked && p.splits == 1 && p.raster_g <= 0 && !STRIDED;
        int c_mu = 0, c_nt = 0, c_wt = 0, c_ht = 0, c_bt = 0;
        for (int item = first_item; ok && item < item_end; item += item_step) {
          int mu, nt, split;
          int w0 = 0, h0 = 0, b0 = 0, tap_n = 0, ci0 = 0;
          Phase phq = {0, 0, p.R, p.S};
          if (stepped) {
            if (item == first_item) {
              decode_item(p, item, c_mu, c_nt, split);
              const int mt0 = c_mu * CTAS + (int)rank;
              tile_coords(p, (IC) ? mt0 * BM : mt0, c_wt, c_ht, c_bt);
            } else if (++c_nt == p.n_tiles_n) {
              c_nt = 0;
              ++c_mu;
              if (IC) {
                tile_coords(p, (c_mu * CTAS + (int)rank) * BM, c_wt, c_ht, c_bt);
              } else {
                c_wt += CTAS;
                while (c_wt >= p.w_tiles) { c_wt -= p.w_tiles; if (++c_ht == p.h_tiles) { c_ht = 0; ++c_bt; } }
              }
            }
            mu = c_mu; nt = c_nt; split = 0;
            w0 = c_wt * p.Wt; h0 = c_ht * p.Ht; b0 = c_bt * p.Bt;
          } else {
            int tile = item;
            if (STRIDED) phq = split_phase(p, item, tile);
            decode_item(p, tile, mu, nt, split);
            if (KIND == GK_CONV_FWD || KIND == GK_CONV_DGRAD)
              pixel_box(p, (mu * CTAS + (int)rank) * ((IC) ? BM : 1), w0, h0, b0);
          }
          if (KIND == GK_CONV_FWD) { w0 *= p.stride_w; h0 *= p.stride; }     // output pixel -> window origin in x
          if (IC) { w0 += p.i2c_w0; h0 += p.i2c_h0; }
          const int n_ts = phq.n_s;
          const int mt = mu * CTAS + (int)rank;     // this CTA's 128-row tile
          const int nb = nt * p.bn + (int)rank * bn_cta;
          const int kb0 = split * p.kb_per_split;
          int kb1 = kb0 + p.kb_per_split;
          if (kb1 > p.kb_total) kb1 = p.kb_total;
          if (STRIDED) kb1 = phq.n_r * phq.n_s * p.c_chunks;
          if (KIND == GK_CONV_WGRAD) {
            if (p.tg > 1) {
              tap_n = nt * p.tg + (int)rank * (p.tg / CTAS);
            } else {
              tap_n = div_by(nt, p.d_chunks);
              ci0 = (nt - tap_n * p.n_chunks) * p.bn + (int)rank * bn_cta;
            }
          }
          // k-block counters, stepped instead of divided inside the loop (one thread issues all copies,
          // so every scalar instruction here is on the critical path):
          //   forward / dgrad: k-block = (tap row r, tap column s, channel chunk cc)
          //   wgrad:           k-block = pixel box (kwt, kht, kbt)
          int cc = 0, ts = 0, tr = 0, kwt = 0, kht = 0, kbt = 0;
          if (kb0 != 0) {
            if (KIND == GK_CONV_FWD || KIND == GK_CONV_DGRAD) {
              const int tap = div_by(kb0, p.d_cc);
              cc = kb0 - tap * p.c_chunks; tr = div_by(tap, p.d_S); ts = tap - tr * p.S;
            } else if (KIND == GK_CONV_WGRAD) {
              tile_coords(p, (IC) ? kb0 * BM : kb0, kwt, kht, kbt);
            }
          }
          int wg_r = 0, wg_s = 0;
          if (KIND == GK_CONV_WGRAD) {
            if (tap_n >= p.R * p.S) tap_n = p.R * p.S - 1;          // (filler of a last, short tap group)
            wg_r = div_by(tap_n, p.d_S); wg_s = tap_n - wg_r * p.S;
          }
          const bool with_b = !resident || item == first_item;       // (resident: the first tile's copies bring them)
          const unsigned tx_bytes = (unsigned)(CTAS * (p.a_boxes * p.a_box_bytes + (with_b ? p.b_boxes * p.b_box_bytes : 0)));
          for (int kb = kb0; kb < kb1; ++kb) {
           if (owner == warp) {
            if (!mbar_wait_warp(empty0 + 8 * stage, phase ^ 1, &abort_flag, status)) { ok = false; break; }
            const unsigned full = lead_full0 + 8 * stage;
            const unsigned sa = smem_base + p.b_res_bytes + stage * stage_bytes;
            const unsigned sb = resident ? smem_base + kb * p.b_tile_bytes : sa + p.a_bytes;
            if (leader) {
            if (rank == 0) mbar_expect_tx(full0 + 8 * stage, tx_bytes);
            switch (KIND) {                       // (one case per instance of the loop)
              case GK_FC_FWD:       // A [M][K] K-major, B [N][K] K-major
                for (int j = 0; j < p.mrep; ++j)     // rows past the end of A are zero-filled by the copy
                  load2<CTAS>(sa + j * p.a_box_bytes, &map_a, full, kb * p.kdepth, (mt * p.mrep + j) * BM);
                if (with_b) load_b(sb, full, kb, 0, 0, nb);
                break;
              case GK_FC_DGRAD:     // A = e [M][N] K-major; B(k', n) = w[n][k'] MN-major
                load2<CTAS>(sa, &map_a, full, kb * p.kdepth, mt * BM);
                if (with_b) load_b(sb, full, kb, 0, 0, nb);
                break;
              case GK_FC_WGRAD:     // A(n, m) = e[m][n] MN-major; B(k', m) = a[m][k'] MN-major
                for (int j = 0; j < p.a_boxes; ++j)
                  load2<CTAS>(sa + j * p.a_box_bytes, &map_a, full, mt * BM + j * p.a_box_step, kb * p.kdepth);
                for (int j = 0; j < p.b_boxes; ++j)
                  load2<CTAS>(sb + j * p.b_box_bytes, &map_b, full, nb + j * p.b_box_step, kb * p.kdepth);
                break;
              case GK_CONV_FWD:     // k-block = (tap, channel chunk); B = w[co][tap][ci]
                if (IC) load_im2col<CTAS>(sa, &map_a, full, cc * p.kdepth, w0, h0, b0, ts, tr);
                else load4<CTAS>(sa, &map_a, full, cc * p.kdepth, w0 + ts - p.pad, h0 + tr - p.pad, b0);
                if (with_b) load_b(sb, full, kb, cc, tr * p.S + ts, nb);
                break;
              case GK_CONV_DGRAD: { // A = e shifted the other way; B(ci, (tap, co)) = w[co][tap][ci]
                int tap = tr * p.S + ts;
                if (IC) {
                  load_im2col<CTAS>(sa, &map_a, full, cc * p.kdepth, w0, h0, b0, p.T_s - 1 - ts, p.T_r - 1 - tr);
                  if (STRIDED) tap = (phq.r + p.dstride * tr) * p.S + phq.s + p.dstride * ts;
                } else {
                  load4<CTAS>(sa, &map_a, full, cc * p.kdepth, w0 - ts + p.pad, h0 - tr + p.pad, b0);
                }
                if (with_b) load_b(sb, full, kb, cc, tap, nb);
                break;
              }
              default: {            // GK_CONV_WGRAD: k-block = pixel box; A = e, B = x shifted by the tap
                const int kw0 = kwt * p.Wt, kh0 = kht * p.Ht, kbb0 = kbt * p.Bt;
                if (IC) {        // consecutive pixels: e as a plain matrix, x as im2col rows of the same pixels
                  for (int j = 0; j < p.a_boxes; ++j)
                    load2<CTAS>(sa + j * p.a_box_bytes, &map_a, full, mt * BM + j * p.a_box_step, kb * BM);
                  for (int j = 0, jb = 0, tr2 = wg_r, ts2 = wg_s; j < p.b_boxes; ++j) {
                    load_im2col<CTAS>(sb + j * p.b_box_bytes, &map_b, full, ci0 + jb * p.b_box_step,
                                      kwt * p.stride_w + p.i2c_w0, kht * p.stride + p.i2c_h0, kbt, ts2, tr2);
                    if (++jb == p.tg_boxes) next_tap(p, jb, tr2, ts2);
                  }
                } else {
                  for (int j = 0; j < p.a_boxes; ++j)
                    load4<CTAS>(sa + j * p.a_box_bytes, &map_a, full, mt * BM + j * p.a_box_step, kw0, kh0, kbb0);
                  for (int j = 0, jb = 0, tr2 = wg_r, ts2 = wg_s; j < p.b_boxes; ++j) {
                    load4<CTAS>(sb + j * p.b_box_bytes, &map_b, full, ci0 + jb * p.b_box_step, kw0 * p.stride + ts2 - p.pad,
                                kh0 * p.stride + tr2 - p.pad, kbb0);
                    if (++jb == p.tg_boxes) next_tap(p, jb, tr2, ts2);
                  }
                }
                break;
              }
            }
            }
           }
            if (KIND == GK_CONV_FWD || KIND == GK_CONV_DGRAD) {
              if (++cc == p.c_chunks) { cc = 0; if (++ts == n_ts) { ts = 0; ++tr; } }
            } else if (KIND == GK_CONV_WGRAD) {
              if (IC) {          // 128 pixels further in the grid
                kwt += p.i2c_dj;
                if (kwt >= p.w_tiles) { kwt -= p.w_tiles; ++kht; }
                kht += p.i2c_di;
                if (kht >= p.h_tiles) { kht -= p.h_tiles; ++kbt; }
                kbt += p.i2c_db;
              } else if (++kwt == p.w_tiles) { kwt = 0; if (++kht == p.h_tiles) { kht = 0; ++kbt; } }
            }
            if (++owner == nprod) owner = 0;
            if (++stage == p.stages) { stage = 0; phase ^= 1; }
          }
        }
      };
      if (ok && first_item < item_end) {
        auto run = [&](auto kind_c) {
          if (I2C && p.i2c) produce(kind_c, std::integral_constant<bool, I2C>{});
          else if (!STRIDED) produce(kind_c, std::false_type{});
        };
        if (STRIDED || p.kind == GK_CONV_DGRAD) run(std::integral_constant<int, GK_CONV_DGRAD>{});
        else if (p.kind == GK_CONV_FWD) run(std::integral_constant<int, GK_CONV_FWD>{});
        else if (p.kind == GK_CONV_WGRAD) run(std::integral_constant<int, GK_CONV_WGRAD>{});
        else if (p.kind == GK_FC_FWD) produce(std::integral_constant<int, GK_FC_FWD>{}, std::false_type{});
        else if (p.kind == GK_FC_DGRAD) produce(std::integral_constant<int, GK_FC_DGRAD>{}, std::false_type{});
        else produce(std::integral_constant<int, GK_FC_WGRAD>{}, std::false_type{});
      }
    }
  } else if (warp == MMA_WARP) {
    // ================= MMA issuer (leader CTA only) =================
    // The whole warp runs the loops in lock step and one elected lane issues: with warp-uniform
    // control flow the descriptor arithmetic stays in the uniform datapath that feeds tcgen05.mma.
    if (rank == 0) {
      const bool leader = elect_one();
      int stage = 0;
      unsigned phase = 0;
      unsigned use = 0;                 // tiles processed by this CTA (pair)
      bool ok = true;
      if (p.halo == 2) {
        // tap pairs (0,1) (2,3) (4,5) (6,7) (8,-): patch row of the first tap and the row distance to
        // the second one (the leading-dimension stride between the two 64-channel halves of M)
        const unsigned a_hi = (unsigned)(p.a_desc >> 32), b_hi = (unsigned)(p.b_desc >> 32);
        const unsigned b_lo0 = (unsigned)p.b_desc;
        unsigned a_pair[5];
#pragma unroll
        for (int pi = 0; pi < 5; ++pi) {
          const int ta = 2 * pi, tb = 2 * pi + 1 < 9 ? 2 * pi + 1 : 2 * pi - 1;
          const int ra = (ta / 3) * 10 + ta % 3, rb = (tb / 3) * 10 + tb % 3;
          const int lbo_rows = rb > ra ? rb - ra : 1;
          a_pair[pi] = (unsigned)(ra * 4) | ((unsigned)(lbo_rows * 4) << 16);     // 64-byte rows, 16-byte units
        }
        for (int item = first_item; ok && item < item_end; item += item_step, ++use) {
          const int split = item - div_by(item, p.d_split) * p.splits;
          const int t0 = split * p.kb_per_split;
          int t1 = t0 + p.kb_per_split;
          if (t1 > p.kb_total) t1 = p.kb_total;
          if (!mbar_wait_warp(tempty0, (use & 1u) ^ 1u, &abort_flag, status)) { ok = false; break; }
          tc_fence_after();
          for (int t = t0; t < t1; ++t) {
            if (!mbar_wait_warp(full0 + 8 * stage, phase, &abort_flag, status)) { ok = false; break; }
            tc_fence_after();
            const unsigned sa16 = ((smem_base + stage * stage_bytes) >> 4) & 0x3fff;
            const unsigned sb16 = ((smem_base + stage * stage_bytes + p.a_bytes) >> 4) & 0x3fff;
            const unsigned first = t > t0 ? 1u : 0u;
            if (leader) {
#pragma unroll
              for (int pi = 0; pi < 5; ++pi) {
#pragma unroll
                for (int j = 0; j < 4; ++j)      // 32 pixels = four rows of eight per MMA
                  tc_mma_i8_lh(tmem_base + 64u * pi, sa16 + a_pair[pi] + 160u * j, a_hi, b_lo0 + sb16 + 128u * j, b_hi,
                               p.idesc, j > 0 ? 1u : first);
              }
              tc_commit(empty0 + 8 * stage);
            }
            if (++stage == p.stages) { stage = 0; phase ^= 1; }
          }
          if (ok && leader) tc_commit(tfull0);
        }
        item_end = first_item;
      } else if (p.halo) {
        halo_mma_loop(p, 0, p.nissue, first_item, item_end, smem_base, tmem_base, full0, empty0, tfull0, tempty0,
                      bres_bar, &abort_flag, status);
        item_end = first_item;
      }
      // generic loop: everything an MMA needs that does not change is read into registers here
      const unsigned g_a_lo0 = (unsigned)p.a_desc, g_b_lo0 = (unsigned)p.b_desc;
      const unsigned g_a_hi = (unsigned)(p.a_desc >> 32), g_b_hi = (unsigned)(p.b_desc >> 32);
      const unsigned g_ak = p.a_kstep16, g_bk = p.b_kstep16, g_idesc = p.idesc, g_a_bytes = (unsigned)p.a_bytes;
      const int g_ksteps = p.ksteps, g_mrep = p.mrep, g_tail = GENERAL ? p.tail_ks : 0;
      const unsigned g_bn_mma = (unsigned)p.bn_mma, g_slice16 = (unsigned)p.a_box_bytes >> 4;
      unsigned gbuf = 0, gpar = 0;            // use % nbuf, (use / nbuf) & 1, counted
      const bool resident = CTAS == 1 && !ONE && !STRIDED && p.b_resident != 0;
      const unsigned g_btile16 = (unsigned)p.b_tile_bytes >> 4;
      for (int item = first_item; ok && item < item_end; item += item_step, ++use) {
        const int split = p.splits > 1 ? item - div_by(item, p.d_split) * p.splits : 0;
        const int kb0 = split * p.kb_per_split;
        int kb1 = kb0 + p.kb_per_split;
        if (kb1 > p.kb_total) kb1 = p.kb_total;
        if (STRIDED) {
          int tile;
          const Phase q = split_phase(p, item, tile);
          kb1 = q.n_r * q.n_s * p.c_chunks;
        }
        int cc_left = g_tail ? p.c_chunks - (kb0 - div_by(kb0, p.d_cc) * p.c_chunks) : 0;     // chunks up to the short one (counted)
        const unsigned buf = gbuf;
        // wait until the epilogue has drained this accumulator buffer (the first nbuf uses pass at once)
        if (!mbar_wait_warp(tempty0 + 8 * buf, gpar ^ 1u, &abort_flag, status)) { ok = false; break; }
        if (++gbuf == (unsigned)p.nbuf) { gbuf = 0; gpar ^= 1u; }
        tc_fence_after();
        const unsigned tmem_d = tmem_base + buf * (unsigned)p.bn;
        for (int kb = kb0; kb < kb1; ++kb) {
          if (!mbar_wait_warp(full0 + 8 * stage, phase, &abort_flag, status)) { ok = false; break; }
          tc_fence_after();
          const unsigned sa = smem_base + p.b_res_bytes + stage * stage_bytes;
          const unsigned a_lo = g_a_lo0 + ((sa >> 4) & 0x3fff);
          const unsigned b_lo = g_b_lo0 + (resident ? ((smem_base >> 4) & 0x3fff) + (unsigned)kb * g_btile16 : ((sa + g_a_bytes) >> 4) & 0x3fff);
          const unsigned first_acc = kb > kb0 ? 1u : 0u;
          int ks = g_ksteps;
          if (g_tail && --cc_left == 0) { ks = g_tail; cc_left = p.c_chunks; }
          if (leader) {
            if (g_mrep > 1) {
              for (int j = 0; j < g_mrep; ++j) {
                const unsigned td = tmem_d + (unsigned)j * g_bn_mma, aj = a_lo + (unsigned)j * g_slice16;
                if (g_ksteps == 1) issue_kblock<CTAS, 1>(td, aj, g_a_hi, b_lo, g_b_hi, g_ak, g_bk, g_idesc, first_acc);
                else if (g_ksteps == 2) issue_kblock<CTAS, 2>(td, aj, g_a_hi, b_lo, g_b_hi, g_ak, g_bk, g_idesc, first_acc);
                else if (g_ksteps == 4) issue_kblock<CTAS, 4>(td, aj, g_a_hi, b_lo, g_b_hi, g_ak, g_bk, g_idesc, first_acc);
                else issue_kblock<CTAS, 3>(td, aj, g_a_hi, b_lo, g_b_hi, g_ak, g_bk, g_idesc, first_acc);
              }
            }
            else if (ks == 4) issue_kblock<CTAS, 4>(tmem_d, a_lo, g_a_hi, b_lo, g_b_hi, g_ak, g_bk, g_idesc, first_acc);
            else if (ks == 2) issue_kblock<CTAS, 2>(tmem_d, a_lo, g_a_hi, b_lo, g_b_hi, g_ak, g_bk, g_idesc, first_acc);
            else if (ks == 1) issue_kblock<CTAS, 1>(tmem_d, a_lo, g_a_hi, b_lo, g_b_hi, g_ak, g_bk, g_idesc, first_acc);
            else issue_kblock<CTAS, 3>(tmem_d, a_lo, g_a_hi, b_lo, g_b_hi, g_ak, g_bk, g_idesc, first_acc);
            // frees the stage (in every CTA of the pair) once these MMAs have read it
            if (CTAS == 2) tc_commit_pair(empty0 + 8 * stage); else tc_commit(empty0 + 8 * stage);
          }
          if (++stage == p.stages) { stage = 0; phase ^= 1; }
        }
        if (ok && leader) {                     // accumulator complete
          if (CTAS == 2) tc_commit_pair(tfull0 + 8 * buf); else tc_commit(tfull0 + 8 * buf);
        }
      }
    }
    if (ONE) {
      // Every CTA has one tile: the sample is the whole tensor, and the shift is exact.  This warp has nothing else to do and
      // speaks for its CTA as soon as the epilogue's warps have reported.
      const long long t0 = clock64();
      while (__any_sync(0xffffffffu, *(volatile unsigned *)&first_arrived < (unsigned)epi_active)) {
        if (__any_sync(0xffffffffu, abort_flag != 0)) break;
        if (__any_sync(0xffffffffu, clock64() - t0 > WAIT_LIMIT_CYCLES)) {
          abort_flag = 1;
          atomicOr(status, NITI_DEV_TIMEOUT);
          break;
        }
      }
      if (__all_sync(0xffffffffu, abort_flag == 0)) {
        unsigned *words = niti_split_max(hdr);
        const int b = (int)niti_agree_bits(words, words + NITI_AGREE_MAX, niti_bitlen32(*(volatile unsigned *)&first_max),
                                           (int)blockIdx.x, (int)gridDim.x, 0, lane, p.patience) - 1;
        if (lane == 0) {
          spec_bp_ready = b < 0 ? -1 : (b > p.mbits ? b - p.mbits : 0) + 1;
          if (b >= 0 && blockIdx.x == 0) publish_exact(b);
        }
      }
    }
  } else if (epi_warp) {
    // ================= epilogue: TMEM -> int32 accumulators + max magnitude =================
    const int quarter = warp & 3;               // TMEM lanes [32 * quarter, +32)
    const int wq = (warp - EPI_WARP0) >> 2;     // index among the four warps of this quarter
    const int egroup = wq >> p.k_wpq_shift;                // tiles use % egroups == egroup are this warp's
    const int chunk_phase = wq & (wpq - 1);           // it takes 32-column chunks phase, phase + wpq, ...
    const int row_in_tile = quarter * 32 + lane;
    unsigned mx = 0;
    int bp = 0;
    if (epi_mode == EPI_KNOWN_B) {
      const int b = niti_bitlen32(hdr->maxabs32);
      bp = b > p.mbits ? b - p.mbits : 0;
    }
    bool ok = true;
    const unsigned red_buf = smem_base + (unsigned)p.red_off + (unsigned)(warp - EPI_WARP0) * 4096u;
    if (!ONE && p.halo == 2) {
      unsigned use = 0;
      // lane = (tap of the pair, input channel), column = output channel; partial sums of this
      // CTA's pixel range are added to g32[co][tap][ci]
      const int which = row_in_tile >> 6, ci = row_in_tile & 63;
      for (int item = first_item; ok && item < item_end; item += item_step, ++use) {
        const int blk = div_by(item, p.d_split);
        const int ci0 = (blk % p.wg_nci) * 64, co0 = (blk / p.wg_nci) * 64;
        if (!mbar_wait(tfull0, use & 1u, &abort_flag, status)) { ok = false; break; }
        tc_fence_after();
        unsigned pmx = 0;                       // largest partial-sum magnitude of this item
        for (int job = chunk_phase; job < 10; job += wpq) {
          const int pi = job >> 1, c0 = (job & 1) * 32;
          const int tap = 2 * pi + which;
          int v[32];
          tc_ld32(tmem_base + ((unsigned)(quarter * 32) << 16) + 64u * pi + (unsigned)c0, v);
          if (tap < 9) {                        // (a warp's 32 rows belong to one tap)
#pragma unroll
            for (int j = 0; j < 32; ++j) pmx = max(pmx, (unsigned)abs(v[j]));
            if (lane == 0) tma_reduce_wait_read();
            __syncwarp();
            stage_tile32<true>(red_buf, lane, v);
            fence_async_shared();
            __syncwarp();
            if (lane == 0) tma_reduce_add_4d(&map_c, red_buf, ci0 + (ci & ~31), tap, co0 + c0, 0);
          }
        }
        pmx = __reduce_max_sync(0xffffffffu, pmx);
        tc_fence_before();
        __syncwarp();
        if (lane == 0) {
          if (pmx) atomicMax(niti_split_max(hdr) + item - blk * p.splits, pmx);
          mbar_arrive(tempty0);
        }
      }
      item_end = first_item;
    }
    const bool fused = epi_mode == EPI_KNOWN_B || epi_mode == EPI_SPECULATE;
    bool unaligned_bp = false;                   // binary point above 24: the lean loop leaves the items to the general one
    // (this warp's staging buffer for rows that are not 32-byte aligned)
    auto nstg = [&]() {
      return reinterpret_cast<unsigned *>(smem_raw + (smem_base - smem_u32(smem_raw)) + p.nstg_off) + (warp - EPI_WARP0) * (32 * 9);
    };
    // this thread's pixel inside a pixel box (generic convolutions): the box sides are powers of two
    struct BoxPixel { int w, h, b; };
    auto box_pixel = [&]() {
      const int t = row_in_tile >> p.wt_shift;
      return BoxPixel{row_in_tile & ((1 << p.wt_shift) - 1), t & ((1 << p.ht_shift) - 1), t >> p.ht_shift};
    };
    // an item's tile: this thread's output row (row-batched mode: in the first of the item's mrep tiles), first column,
    // columns inside the matrix
    struct Tile {
      int mt, nt, split, ncols_valid, out_row, col0;
      bool row_ok;
    };
    auto tile_of = [&](int item) {
      Tile t = {0, 0, 0, 0, 0, 0, false};
      Phase phq = {0, 0, 1, 1};
      int mu = 0;
      if (!p.halo) {
        int tile = item;
        if (STRIDED) phq = split_phase(p, item, tile);
        decode_item(p, tile, mu, t.nt, t.split);
      }
      t.mt = mu * CTAS + (int)rank;
      t.col0 = t.nt * p.bn;
      t.ncols_valid = min(p.gn - t.col0, p.bn);
      if (p.halo) {
        int wt, ht, bt;
        tile_coords(p, item, wt, ht, bt);
        const int w = wt * 8 + (row_in_tile & 7), h = ht * 16 + (row_in_tile >> 3);
        t.row_ok = w < p.PW && h < p.PH;
        t.out_row = (bt * p.PH + h) * p.PW + w;
      } else if (STRIDED) {
        t.out_row = phase_row(p, t.mt * BM + row_in_tile, phq, t.row_ok);
      } else if ((p.kind == GK_CONV_FWD || p.kind == GK_CONV_DGRAD) && !(I2C && p.i2c)) {
        int w0, h0, b0;
        pixel_box(p, t.mt, w0, h0, b0);
        const BoxPixel px = box_pixel();
        const int w = w0 + px.w, h = h0 + px.h, b = b0 + px.b;
        t.row_ok = w < p.PW && h < p.PH && b < p.PB;
        t.out_row = (b * p.PH + h) * p.PW + w;
      } else {
        t.out_row = t.mt * (BM * p.mrep) + row_in_tile;
        t.row_ok = t.out_row < p.gm;
        if (p.kind == GK_CONV_WGRAD) {
          const int tap = div_by(t.nt, p.d_chunks), ci0 = (t.nt - tap * p.n_chunks) * p.bn;
          t.col0 = tap * p.Cn + ci0;
          t.ncols_valid = p.Cn - ci0 < p.bn && p.tg <= 1 ? p.Cn - ci0 : p.bn;
        }
      }
      return t;
    };
    // The first tile of this CTA has largest magnitude m0 in this warp's share.  The warps combine their maxima in shared
    // memory; one warp speaks for the CTA in the grid-wide agreement (with every warp of every CTA polling the same word the
    // wait itself took microseconds) and publishes the shift to the others through shared memory: the issuing warp, idle by
    // then, in single-wave launches, else the last one to report, for which this is true.
    auto report = [&](unsigned m0) {
      m0 = __reduce_max_sync(0xffffffffu, m0);
      unsigned last = 0;
      if (lane == 0) {
        if (m0) atomicMax(&first_max, m0);
        __threadfence_block();
        last = atomicAdd(&first_arrived, 1u) + 1u == (unsigned)epi_active ? 1u : 0u;
      }
      if (ONE) return false;
      if (!__shfl_sync(0xffffffffu, last, 0)) return false;
      const int b = agree_on_guess(hdr, *(volatile unsigned *)&first_max, p.patience, p.spec_mul256, p.spec_tag, spec_slot, lane);
      if (lane == 0) {
        cta_b = b;
        spec_bp_ready = (b > p.mbits ? b - p.mbits : 0) + 1;
      }
      return true;
    };
    // What this CTA's first tile alone says about the tensor's binary point, once all its warps have reported.
    auto own_guess = [&]() {
      const long long t0 = clock64();
      while (*(volatile unsigned *)&first_arrived < (unsigned)epi_active && !abort_flag && clock64() - t0 < WAIT_LIMIT_CYCLES) {
      }
      __syncwarp();
      const unsigned own = *(volatile unsigned *)&first_max;
      const unsigned long long scaled = ((unsigned long long)own * p.trial_mul256) >> 8;
      const int b = niti_bitlen32(scaled > 0x7fffffffull ? 0x7fffffffu : (unsigned)scaled);
      return __shfl_sync(0xffffffffu, b > p.mbits ? b - p.mbits : 0, 0);
    };
    // The agreed binary point (in spec_bp_ready), once it is there; false: time to leave.
    auto await_bp = [&]() {
      if (lane == 0) {
        const long long t1 = clock64();
        while (spec_bp_ready == 0) {
          if (abort_flag) break;
          if (clock64() - t1 > WAIT_LIMIT_CYCLES) {
            abort_flag = 1;
            atomicOr(status, NITI_DEV_TIMEOUT);
            break;
          }
        }
      }
      __syncwarp();
      return abort_flag == 0;
    };
    // ---- lean loop: fused rounding (every layer of the networks) ----
    // The epilogue warps share their schedulers' integer pipe with everything else, and with few
    // input channels that pipe is the bound of the whole kernel: per tile and per chunk this loop
    // executes only what changes (measured on the first layer: a loop that tests the launch's options per tile and
    // chunk spends a third of its integer instructions on tests whose outcome is the same for every tile).
    // Code that is not in the SM's instruction cache costs about 8 ns an instruction (lines of 128 bytes, 70 - 100 ns each), and
    // in a program of different kernels that is every launch: rounding the first tile took 4.3 us instead of the 1.9 us of a
    // launch that repeats.  While the bit-width is being agreed (2 us), the warps therefore round and store the first tile
    // with what the tile itself says of the bit-width (`trial`), and again only where the grid has agreed on another one; where
    // a store could not be taken back (weight updates, outputs in the storage of an operand) a chunk passes without it.
    auto lean_as = [&](auto relu_c, auto mask_c, auto batched_c, auto pool_c, auto upd_c, auto narrow_c) {
      constexpr bool NARROW = decltype(narrow_c)::value;   // output rows that are not 32-byte aligned, short last chunks
      constexpr bool RELU = decltype(relu_c)::value, MASK = decltype(mask_c)::value, BATCHED = decltype(batched_c)::value;
      constexpr bool POOL = decltype(pool_c)::value;       // fused 2 x 2 max-pool of the ReLU'd tile
      constexpr bool UPD = decltype(upd_c)::value;         // the output rows are weights: subtract the rounded gradient
      const int pool_xh = p.pool_xh;
      const bool pool_lane = (lane & (1 | pool_xh)) == 0;  // the window's top-left pixel stores the maximum
      const int kind = STRIDED ? (int)ROWS_PHASES : p.row_kind;
      const int istep = item_step * egroups, nbuf = p.nbuf, bn = p.bn, n_tiles_n = p.n_tiles_n;
      const int cstep = 32 * wpq, c_first = 32 * chunk_phase;
      const int gn = p.gn, gm = p.gm;
      const int bn_mma = BATCHED ? p.bn_mma : p.bn;
      const bool counted = p.blocked && p.raster_g <= 0 && kind != ROWS_PHASES;     // consecutive items: (mu, nt) are stepped
      const int lean_item = first_item + egroup * item_step;
      unsigned ebuf = (unsigned)egroup, epar = 0;           // use % nbuf, (use / nbuf) & 1 (nbuf is a multiple of egroups)
      Extremes ex_all = {0, 0, 0u};
      RoundConst rk = {0u, 0u, 0u, 0, 0, 0u, 0u, 0u, 0u, 0u, true};
      const BoxPixel bpx = box_pixel();
      int mu = 0, nt = 0, split = 0, h_wt = 0, h_ht = 0, h_bt = 0;
      if (epi_mode == EPI_KNOWN_B) {
        rk = make_round_const(bp, p.mbits, p.round_mode);
        if (!rk.aligned) { unaligned_bp = true; return; }
      }
      Phase phq = {0, 0, 1, 1};
      if (kind == ROWS_PHASES) {
        int tile;
        phq = split_phase(p, lean_item, tile);
        decode_item(p, tile, mu, nt, split);
      } else if (kind != ROWS_HALO) decode_item(p, lean_item, mu, nt, split);
      else tile_coords(p, lean_item, h_wt, h_ht, h_bt);
      for (int item = lean_item; item < item_end; item += istep) {
        const unsigned buf = ebuf, tpar = epar;
        ebuf += (unsigned)egroups;
        if (ebuf >= (unsigned)nbuf) { ebuf -= (unsigned)nbuf; epar ^= 1u; }
        int out_row, pool_row = 0;
        bool row_ok;
        int col0 = nt * bn;
        int cend = BATCHED ? bn : gn - col0;          // (whole chunks unless NARROW)
        if (kind == ROWS_HALO) {
          const int w = h_wt * 8 + (row_in_tile & 7), h = h_ht * 16 + (row_in_tile >> 3);
          row_ok = w < p.PW && h < p.PH;
          out_row = (h_bt * p.PH + h) * p.PW + w;
          if (POOL) pool_row = (h_bt * (p.PH >> 1) + (h >> 1)) * (p.PW >> 1) + (w >> 1);
          h_wt += egroups;
          while (h_wt >= p.w_tiles) { h_wt -= p.w_tiles; if (++h_ht == p.h_tiles) { h_ht = 0; ++h_bt; } }
        } else if (kind == ROWS_BOXES) {
          int w0, h0, b0;
          pixel_box(p, mu * CTAS + (int)rank, w0, h0, b0);
          const int w = w0 + bpx.w, h = h0 + bpx.h, b = b0 + bpx.b;
          row_ok = w < p.PW && h < p.PH && b < p.PB;
          out_row = (b * p.PH + h) * p.PW + w;
          if (POOL) pool_row = (b * (p.PH >> 1) + (h >> 1)) * (p.PW >> 1) + (w >> 1);
        } else if (kind == ROWS_PHASES) {
          out_row = phase_row(p, (mu * CTAS + (int)rank) * BM + row_in_tile, phq, row_ok);
        } else {
          out_row = (mu * CTAS + (int)rank) * (BM * p.mrep) + row_in_tile;
          row_ok = out_row < gm;
          if (kind == ROWS_WGRAD) {
            const int tap = div_by(nt, p.d_chunks), ci0 = (nt - tap * p.n_chunks) * bn;
            col0 = tap * p.Cn + ci0;
            cend = p.Cn - ci0;
          }
        }
        if (cend > bn) cend = bn;
        if (!ONE && kind != ROWS_HALO) {                       // next item of this warp
          if (counted) { nt += egroups; while (nt >= n_tiles_n) { nt -= n_tiles_n; ++mu; } }
          else if (item + istep < item_end) {
            int tile = item + istep;
            if (kind == ROWS_PHASES) phq = split_phase(p, item + istep, tile);
            decode_item(p, tile, mu, nt, split);
          }
        }
        const unsigned tm_row = tmem_base + ((unsigned)(quarter * 32) << 16) + buf * (unsigned)bn;
        int live = 1, ce = cend, trial_bp = -1;                // columns of this pass; the binary point of a trial
        if (epi_mode == EPI_SPECULATE && item == lean_item) {
          live = 0;
          ce = c_first + 1;
          if (egroup == 0) {
            // first tile of this CTA: max only, then agree on the estimate with the whole grid (columns of a partly filled
            // chunk beyond the matrix accumulate zeros; whole chunks beyond it are left out)
            int hi0 = 0, lo0 = 0, t = 0;
            asm volatile("" : "+r"(t));                 // (one copy of the loop: the first, empty pass is for the instruction cache)
#pragma unroll 1
            for (; t < 2; ++t) {
              if (t && !mbar_wait(tfull0 + 8 * buf, tpar, &abort_flag, status)) { ok = false; break; }
              tc_fence_after();
              hi0 = lo0 = 0;
              for (int c = c_first; c < (t ? cend : c_first + 1); c += cstep) {
                int v[32];
                tc_ld32(tm_row + (unsigned)c, v);
                if (row_ok && (!BATCHED || out_row + c / bn_mma * BM < gm)) {
#pragma unroll
                  for (int j = 0; j < 32; j += 2) {
                    hi0 = __vimax3_s32(hi0, v[j], v[j + 1]);
                    lo0 = __vimin3_s32(lo0, v[j], v[j + 1]);
                  }
                }
              }
            }
            if (!ok) break;
            if (report(max((unsigned)hi0, 0u - (unsigned)lo0))) {
              ce = c_first;                                    // (the agreement is there)
            } else if (!UPD && p.trial_mul256) {
              trial_bp = own_guess();
              if (trial_bp <= 24) {
                rk = make_round_const(trial_bp, p.mbits, p.round_mode);
                ce = cend;
              } else {
                trial_bp = -1;
              }
            }
          }
        } else if (!mbar_wait(tfull0 + 8 * buf, tpar, &abort_flag, status)) {
          ok = false;
          break;
        }
        tc_fence_after();
        const unsigned row_off = (unsigned)out_row * (unsigned)gn + (unsigned)col0;       // (used where row_ok)
#pragma unroll 1
        while (true) {
          unsigned off = row_off;                              // (row-batched mode: steps to the item's next 128-row tile)
          int orow = out_row;
          int cc = c_first;
          if (BATCHED) while (cc >= bn_mma) { cc -= bn_mma; orow += BM; off += BM * (unsigned)gn; }
          for (int c = c_first; c < ce; c += cstep) {
            int v[32];
            const bool rok = (BATCHED ? (row_ok && orow < gm) : row_ok) && (live != 0 || trial_bp >= 0);   // (rows that are read and written)
            unsigned m[8];
            if (NARROW) {
              if (MASK && rok) load_row_narrow(mask8 + (off + cc), m, cend - c < 32 ? cend - c : 32);
            } else if ((MASK || UPD) && rok)
              asm volatile("ld.global.v8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                           : "=r"(m[0]), "=r"(m[1]), "=r"(m[2]), "=r"(m[3]), "=r"(m[4]), "=r"(m[5]), "=r"(m[6]), "=r"(m[7])
                           : "l"((UPD ? (const int8_t *)out8 : mask8) + (off + cc)));
            tc_ld32(tm_row + (unsigned)c, v);
            unsigned w8[8];
            if (POOL) {
#pragma unroll
              for (int j = 0; j < 8; ++j) w8[j] = 0u;          // lanes outside the tensor pool zeros
            }
            if (rok || (!live && trial_bp < 0)) {
#pragma unroll
              for (int j = 0; j < 8; ++j) {
                w8[j] = round_pack4_aligned<RELU>(v[4 * j], v[4 * j + 1], v[4 * j + 2], v[4 * j + 3], rk, ex_all);
                if (MASK) w8[j] &= bytes_gt0(m[j]);
                if (UPD) w8[j] = bytes_sub_clamp127(m[j], w8[j]);
              }
              if (!NARROW && rok) store32(out8 + (off + cc), w8);
            }
            if (NARROW) store_rows_narrow(out8, off + cc, rok, w8, BATCHED ? gn - cc : cend - c, p.io_unit, nstg(), lane);
            if (POOL) {                                        // (warp-uniform: all lanes exchange)
              pool_chunk32(w8, pool_xh);
              if (rok && pool_lane) store32(pool8 + ((unsigned)pool_row * (unsigned)gn + (unsigned)(col0 + cc)), w8);
            }
            cc += cstep;
            if (BATCHED) while (cc >= bn_mma) { cc -= bn_mma; orow += BM; off += BM * (unsigned)gn; }
          }
          if (live) break;
          if (!await_bp()) { ok = false; break; }
          if (ONE && spec_bp_ready < 0) {                      // (this CTA leaves: see niti_agree_bits)
            for (int c = c_first; c < cend; c += cstep) {
              int v[32];
              tc_ld32(tm_row + (unsigned)c, v);
              if (!row_ok) continue;
#pragma unroll
              for (int j = 0; j < 32; ++j)
                if (c + j < cend) acc[row_off + c + j] = v[j];
            }
            ok = false;
            break;
          }
          bp = spec_bp_ready - 1;
          if (bp == trial_bp) break;                           // (stored already)
          trial_bp = -1;
          ce = cend;
          rk = make_round_const(bp, p.mbits, p.round_mode);
          ex_all = Extremes{0, 0, 0u};
          if (!rk.aligned) { unaligned_bp = true; break; }
          if (egroup != 0 && !mbar_wait(tfull0 + 8 * buf, tpar, &abort_flag, status)) { ok = false; break; }
          tc_fence_after();
          live = 1;
          asm volatile("" : "+r"(live));                       // (one copy of the loop)
        }
        if (ONE || !ok || unaligned_bp) break;
        tc_fence_before();
        __syncwarp();
        if (lane == 0) {
          if (CTAS == 2 && rank != 0) mbar_arrive_cluster(lead_tempty0 + 8 * buf);
          else mbar_arrive(tempty0 + 8 * buf);
        }
      }
      mx |= ex_all.magnitude_bits();
    };
    auto lean = [&]() __attribute__((always_inline)) {
      using T = std::true_type;
      using F = std::false_type;
      const int form = p.form;
      if (form == LEAN_RELU) lean_as(T{}, F{}, F{}, F{}, F{}, F{});
      else if (form == LEAN_MASK) lean_as(F{}, T{}, F{}, F{}, F{}, F{});
      else if (form == LEAN_POOL) lean_as(T{}, F{}, F{}, T{}, F{}, F{});
      else if (form == LEAN_PLAIN) lean_as(F{}, F{}, F{}, F{}, F{}, F{});
      else if (form == LEAN_UPDATE) lean_as(F{}, F{}, F{}, F{}, T{}, F{});
      else if (GENERAL && form == LEAN_NARROW_RELU) lean_as(T{}, F{}, F{}, F{}, F{}, T{});
      else if (GENERAL && form == LEAN_NARROW_MASK) lean_as(F{}, T{}, F{}, F{}, F{}, T{});
      else if (GENERAL && form == LEAN_NARROW) lean_as(F{}, F{}, F{}, F{}, F{}, T{});
      else if (!ONE && form == LEAN_BATCHED_RELU) lean_as(T{}, F{}, T{}, F{}, F{}, F{});
      else if (!ONE && form == LEAN_BATCHED) lean_as(F{}, F{}, T{}, F{}, F{}, F{});
      else if (!ONE && GENERAL && form == LEAN_BATCHED_NARROW_RELU) lean_as(T{}, F{}, T{}, F{}, F{}, T{});
      else if (!ONE && GENERAL && form == LEAN_BATCHED_NARROW) lean_as(F{}, F{}, T{}, F{}, F{}, T{});
    };
    // ---- the loop for everything else: accumulators kept, partial sums, rounding that the lean loop does not do ----
    auto general = [&]() {
      unsigned use = (unsigned)egroup, ebuf = (unsigned)egroup, epar = 0;
      const RoundConst rk = make_round_const(bp, p.mbits, p.round_mode);
      for (int item = first_item + egroup * item_step; ok && item < item_end;
           item += item_step * egroups, use += (unsigned)egroups) {
        const Tile t = tile_of(item);
        const int mt = t.mt, nt = t.nt, split = t.split, ncols_valid = t.ncols_valid;
        const int out_row = t.out_row, col0 = t.col0;
        const bool row_ok = t.row_ok;
        const unsigned buf = ebuf;
        const unsigned tpar = epar;
        ebuf += (unsigned)egroups;
        if (ebuf >= (unsigned)p.nbuf) { ebuf -= (unsigned)p.nbuf; epar ^= 1u; }
        if (!mbar_wait(tfull0 + 8 * buf, tpar, &abort_flag, status)) { ok = false; break; }
        tc_fence_after();
        const unsigned tm_row = tmem_base + ((unsigned)(quarter * 32) << 16) + buf * (unsigned)p.bn;
        if (epi_mode == EPI_ATOMIC && p.red) {
          // partial sums of a split contraction: every chunk is staged and added by one copy
          unsigned pmx = 0;                                      // largest partial-sum magnitude of this item
          int x0, x1, x2 = 0, x3 = 0;                            // tensor coordinates of the chunk at column 0
          if (p.kind == GK_CONV_WGRAD) {
            const int tap = div_by(nt, p.d_chunks);
            x0 = (nt - tap * p.n_chunks) * p.bn;
            x1 = tap;
            x2 = mt * BM + quarter * 32;
          } else if (p.red == 2) {                               // pixel boxes
            x0 = (int)col0;
            int w0, h0, b0;
            pixel_box(p, mt, w0, h0, b0);
            const BoxPixel px = box_pixel();
            x1 = __shfl_sync(0xffffffffu, w0 + px.w, 0);
            x2 = __shfl_sync(0xffffffffu, h0 + px.h, 0);
            x3 = __shfl_sync(0xffffffffu, b0 + px.b, 0);
          } else {
            x0 = (int)col0;
            x1 = mt * BM + quarter * 32;
          }
          const bool any_row = __any_sync(0xffffffffu, row_ok);
          for (int c = 32 * chunk_phase; c < p.bn && c < ncols_valid && any_row; c += 32 * wpq) {
            int xc = x0 + c, xt = x1;
            if (p.kind == GK_CONV_WGRAD && p.tg > 1) {           // tap group: tg_cols (a power of two) columns per tap
              xt = nt * p.tg + c / p.tg_cols;
              xc = c & (p.tg_cols - 1);
              if (xt >= p.R * p.S || xc >= p.Cn) continue;
            }
            int v[32];
            tc_ld32(tm_row + (unsigned)c, v);
            // (rows and columns outside the matrix are clipped by the copy; they may hold anything)
            if (row_ok) {
  #pragma unroll
              for (int j = 0; j < 32; ++j) pmx = max(pmx, (unsigned)abs(v[j]));
            }
            if (lane == 0) tma_reduce_wait_read();
            __syncwarp();
            stage_tile32<false>(red_buf, lane, v);
            fence_async_shared();
            __syncwarp();
            if (lane == 0) tma_reduce_add_4d(&map_c, red_buf, xc, xt, x2, x3);
          }
          pmx = __reduce_max_sync(0xffffffffu, pmx);
          if (lane == 0 && pmx) atomicMax(niti_split_max(hdr) + split, pmx);
        } else if (epi_mode <= EPI_ATOMIC) {
          int32_t *dst = acc + ((long long)out_row * p.gn + col0);
          const bool vec_ok = ((p.gn & 3) == 0) && ((col0 & 3) == 0);
          unsigned pmx = 0;                                      // largest partial-sum magnitude of this item
          for (int c = 32 * chunk_phase; c < p.bn; c += 32 * wpq) {
            int v[32];
            tc_ld32(tm_row + (unsigned)c, v);
            if (row_ok && c < ncols_valid) {
              if (epi_mode == EPI_ATOMIC) {
  #pragma unroll
                for (int j = 0; j < 32; ++j)
                  if (c + j < ncols_valid && v[j] != 0) {
                    pmx = max(pmx, (unsigned)abs(v[j]));
                    atomicAdd(dst + c + j, v[j]);
                  }
              } else {
                if (vec_ok && c + 32 <= ncols_valid) {
  #pragma unroll
                  for (int j = 0; j < 32; j += 4) {
                    *reinterpret_cast<int4 *>(dst + c + j) = make_int4(v[j], v[j + 1], v[j + 2], v[j + 3]);
                  }
  #pragma unroll
                  for (int j = 0; j < 32; ++j) {
                    unsigned a = v[j] < 0 ? 0u - (unsigned)v[j] : (unsigned)v[j];
                    mx = a > mx ? a : mx;
                  }
                } else {
  #pragma unroll
                  for (int j = 0; j < 32; ++j)
                    if (c + j < ncols_valid) {
                      dst[c + j] = v[j];
                      unsigned a = v[j] < 0 ? 0u - (unsigned)v[j] : (unsigned)v[j];
                      mx = a > mx ? a : mx;
                    }
                }
              }
            }
          }
          if (epi_mode == EPI_ATOMIC) {
            pmx = __reduce_max_sync(0xffffffffu, pmx);
            if (lane == 0 && pmx) atomicMax(niti_split_max(hdr) + split, pmx);
          }
        } else {
          // Whole 32-column chunks with 32-byte aligned rows (binary points above 24), or any rows.
          const bool whole_chunks = p.io_unit == 32;
          for (int c = 32 * chunk_phase; c < p.bn; c += 32 * wpq) {
            // chunk geometry: in row-batched mode chunk c holds columns cc of the item's tile c / bn_mma
            const int jt = p.mrep > 1 ? c / p.bn_mma : 0, cc = c - jt * p.bn_mma;
            const int orow = out_row + jt * BM;
            const unsigned off = (unsigned)orow * (unsigned)p.gn + (unsigned)(col0 + cc);
            const bool rok = row_ok && (p.mrep == 1 || orow < p.gm);
            const int nv = ncols_valid - cc;                     // (uniform across the warp)
            if (nv <= 0) continue;
            // (the bytes of the ReLU mask, or the weights this chunk updates, are fetched first)
            int v[32];
            unsigned m[8], w8[8];
            const int8_t *const src = p.update ? (const int8_t *)out8 : mask8;
            if (src && rok) load_row_narrow(src + off, m, nv < 32 ? nv : 32);
            tc_ld32(tm_row + (unsigned)c, v);
            if (rok) {
              Extremes ex = {0, 0, 0u};                          // (columns beyond the matrix accumulate zeros)
              round_chunk32(v, w8, rk, p.relu != 0, ex);
              mx |= ex.magnitude_bits();
              if (src) {
#pragma unroll
                for (int j = 0; j < 8; ++j) w8[j] = p.update ? bytes_sub_clamp127(m[j], w8[j]) : w8[j] & bytes_gt0(m[j]);
              }
            }
            if (whole_chunks) { if (rok) store32(out8 + off, w8); }
            else if (GENERAL) store_rows_narrow(out8, off, rok, w8, nv, p.io_unit, nstg(), lane);
          }
        }
        tc_fence_before();
        __syncwarp();
        if (lane == 0) {
          if (CTAS == 2 && rank != 0) mbar_arrive_cluster(lead_tempty0 + 8 * buf);
          else mbar_arrive(tempty0 + 8 * buf);
        }
      }
    };
    if (fused) lean();
    if (!fused || unaligned_bp) general();
    if (epi_mode == EPI_SPILL || epi_mode == EPI_SPECULATE) {
      mx = __reduce_max_sync(0xffffffffu, mx);
      if (ONE) {
        // (a CTA that rounded with the agreed bit-width has met nothing wider: anything else means that the agreement was
        // broken and its stored values are not exact)
        if (lane == 0 && spec_bp_ready > 0 && niti_bitlen32(mx) > p.mbits + spec_bp_ready - 1) atomicOr(status, NITI_DEV_INTERNAL);
      } else if (lane == 0 && mx) {
        atomicMax(&cta_max, mx);                        // (one global atomic per CTA, below)
      }
    }
    if (p.red && lane == 0) tma_reduce_wait_all();      // (shared memory stays valid until the copies are done)
  }

  // ================= common exit =================
  tc_fence_before();
  __syncthreads();
  if (!ONE && threadIdx.x == 0) {
    if (cta_max) atomicMax(&hdr->maxabs32, cta_max);
    if (cta_b >= 0) atomicOr(&hdr->spec_mask, 1u << cta_b);
  }
  if (abort_flag) {
    // give copies and MMAs still in flight time to land before shared and tensor memory go away
    long long t0 = clock64();
    while (clock64() - t0 < 20000000LL) {
    }
    __syncthreads();
  } else if (ONE) {
    niti_finish_left(hdr, niti_split_max(hdr), spec_bp_ready < 0, ticket, [&](int j) {
      const unsigned bits = niti_posted_bits(niti_split_max(hdr), (int)gridDim.x, status);
      if (bits == 0) return;
      if (j == 0 && threadIdx.x == 0) publish_exact((int)bits - 1);
      round_left_tile<CTAS, STRIDED>(p, j, (int)bits - 1, acc, out8, mask_at_exit, pool8);
    });
  }
  if (CTAS == 2) cluster_sync_all();   // nobody leaves while the peer may still touch this CTA
  if (warp == MMA_WARP) {
    tc_fence_after();
    if (CTAS == 2)
      asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(tmem_cols) : "memory");
    else
      asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(tmem_cols) : "memory");
  }
}

// Finish of a split contraction in one launch: bit-width of the int32 sums, rounding, ReLU / gate / weight update.  The
// sums stay in registers across the grid-wide agreement (at most one block per SM, NV x 4 values per thread), so they
// are read once.  Bound: latency; as two kernels (maximum, then rounding) the finish of a 64 x 64 x 9 gradient took 5.2
// us and that of a 512 x 512 x 9 one 8.7 us.
constexpr int FIN_THREADS = 512;
template <int NV>
__global__ void __launch_bounds__(FIN_THREADS, 1)
finish_split_kernel(const int32_t *__restrict__ acc, int nvec, WsHeader *hdr, int splits, uint32_t *status, int8_t *out,
                    int8_t *upd, const int8_t *__restrict__ mask, int relu, int mbits, int round_mode, const int32_t *s_a,
                    const int32_t *s_w, int32_t *s_out, int32_t *b_out, unsigned patience) {
  __shared__ unsigned blk_max, agreed, ticket;
  const int tid = (int)threadIdx.x, lane = tid & 31, warp = tid >> 5, T = (int)gridDim.x * FIN_THREADS;
  if (tid == 0) blk_max = 0;
  niti_enter(acc, mask);                                      // the multiply has completed and is visible
  unsigned came = 0;
  if (tid == 64) came = niti_arrive(hdr);
  int4 v[NV];
  auto load = [&](int blk) {
#pragma unroll
    for (int i = 0; i < NV; ++i) {
      const int idx = blk * FIN_THREADS + tid + i * T;
      v[i] = make_int4(0, 0, 0, 0);
      if (idx < nvec) v[i] = __ldcg(reinterpret_cast<const int4 *>(acc) + idx);
    }
  };
  load((int)blockIdx.x);
  unsigned mx = 0;
#pragma unroll
  for (int i = 0; i < NV; ++i) {
    mx = max(mx, max((unsigned)abs(v[i].x), (unsigned)abs(v[i].y)));
    mx = max(mx, max((unsigned)abs(v[i].z), (unsigned)abs(v[i].w)));
  }
  mx = __reduce_max_sync(0xffffffffu, mx);
  __syncthreads();
  if (lane == 0 && mx) atomicMax(&blk_max, mx);
  if (blockIdx.x == 0 && warp == 1) {
    // the largest partial sums of all splits bound every total (int32 range)
    unsigned long long bound = 0;
    for (int i = lane; i < splits; i += 32) bound += niti_split_max(hdr)[i];
    for (int o = 16; o > 0; o >>= 1) bound += __shfl_xor_sync(0xffffffffu, bound, o);
    if (lane == 0 && bound >= 0x80000000ull) atomicOr(status, NITI_DEV_ACC_RANGE);
  }
  __syncthreads();
  // (behind the split maxima: the caller leaves room)
  unsigned *words = niti_split_max(hdr) + NITI_MAX_SPLITS - NITI_AGREE_WORDS;
  if (warp == 0) {
    const unsigned m = niti_agree_bits(words, words + NITI_AGREE_MAX, niti_bitlen32(blk_max), (int)blockIdx.x, (int)gridDim.x, 0, lane,
                                       patience);
    if (lane == 0) agreed = m;
  }
  if (tid == 64) ticket = came;
  __syncthreads();
  auto round_block = [&](int blk, unsigned bits) {
    const int b = (int)bits - 1, bp = b > mbits ? b - mbits : 0;
    if (blk == 0 && tid == 0) {
      if (b_out) *b_out = b;
      if (s_out) {
        const int s = bp + (s_a ? *s_a : 0) + (s_w ? *s_w : 0);
        *s_out = s;
        if (s < -128 || s > 127) atomicOr(status, NITI_DEV_EXP_RANGE);
      }
    }
    const RoundConst rk = make_round_const(bp, mbits, round_mode);
    Extremes ex = {0, 0, 0u};
#pragma unroll
    for (int i = 0; i < NV; ++i) {
      const int idx = blk * FIN_THREADS + tid + i * T;
      if (idx >= nvec) break;
      unsigned w = rk.aligned ? round_pack4_aligned<false>(v[i].x, v[i].y, v[i].z, v[i].w, rk, ex)
                              : round_pack4<false, true>(v[i].x, v[i].y, v[i].z, v[i].w, rk, ex);
      if (relu) w &= bytes_gt0(w);
      if (mask) w &= bytes_gt0(reinterpret_cast<const unsigned *>(mask)[idx]);
      if (upd) reinterpret_cast<unsigned *>(upd)[idx] = bytes_sub_clamp127(reinterpret_cast<unsigned *>(upd)[idx], w);
      else reinterpret_cast<unsigned *>(out)[idx] = w;
    }
  };
  const unsigned got = agreed, came_as = ticket;
  if (got) round_block((int)blockIdx.x, got);
  if (got && !(came_as >> 16)) return;
  // (the sums of a block that left are in memory already)
  niti_finish_left(hdr, words, got == 0, came_as, [&](int j) {
    const unsigned bits = niti_posted_bits(words, (int)gridDim.x, status);
    if (bits == 0) return;
    load(j);
    round_block(j, bits);
  });
}

// Self-test of the bounded wait: one warp waits on a barrier that nothing ever completes, gives up
// after ~50 ms, raises NITI_DEV_TIMEOUT and returns normally (the context stays usable).
__global__ void timeout_probe_kernel(uint32_t *status) {
  __shared__ __align__(8) unsigned long long bar;
  __shared__ volatile int abort_flag;
  if (threadIdx.x == 0) {
    abort_flag = 0;
    mbar_init(smem_u32(&bar), 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncthreads();
  if (threadIdx.x == 0) (void)mbar_wait(smem_u32(&bar), 0, &abort_flag, status, 100000000LL);
  __syncthreads();
}

// ------------------------------------------------------------------------------------------
// Host side: tensor maps, descriptors, eligibility
// ------------------------------------------------------------------------------------------
typedef CUresult (*EncodeIm2colFn)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *, const cuuint64_t *,
                                   const cuuint64_t *, const int *, const int *, cuuint32_t, cuuint32_t,
                                   const cuuint32_t *, CUtensorMapInterleave, CUtensorMapSwizzle,
                                   CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
typedef CUresult (*EncodeTiledFn)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *, const cuuint64_t *,
                                  const cuuint64_t *, const cuuint32_t *, const cuuint32_t *,
                                  CUtensorMapInterleave, CUtensorMapSwizzle, CUtensorMapL2promotion,
                                  CUtensorMapFloatOOBfill);

static CUtensorMapSwizzle swizzle_enum(int bytes) {
  return bytes == 128 ? CU_TENSOR_MAP_SWIZZLE_128B : (bytes == 64 ? CU_TENSOR_MAP_SWIZZLE_64B : CU_TENSOR_MAP_SWIZZLE_32B);
}
static unsigned long long layout_bits(int swizzle_bytes) {
  // matrix-descriptor layout type: 2 = 128-byte swizzle, 4 = 64-byte, 6 = 32-byte
  unsigned long long t = swizzle_bytes == 128 ? 2 : (swizzle_bytes == 64 ? 4 : 6);
  return t << 61;
}
// Descriptor (without start address) of a K-major operand whose rows are `sw` bytes wide.
static unsigned long long desc_kmajor(int sw, int group_rows = 8) {
  unsigned long long d = 0;
  d |= (unsigned long long)1 << 16;                          // leading byte offset: unused, 1
  d |= (unsigned long long)((group_rows * sw) >> 4) << 32;   // stride between 8-row groups
  d |= (unsigned long long)1 << 46;                          // descriptor version
  return d | layout_bits(sw);
}
// Descriptor of an MN-major operand stored as sub-tiles [kdepth rows][sw bytes].
static unsigned long long desc_mnmajor(int sw, int kdepth) {
  unsigned long long d = 0;
  d |= (unsigned long long)((kdepth * sw) >> 4) << 16;       // next sw-wide chunk along M/N
  d |= (unsigned long long)((8 * sw) >> 4) << 32;            // next group of 8 k-rows
  d |= (unsigned long long)1 << 46;
  return d | layout_bits(sw);
}
// Swizzle width (= bytes of a copied row) of an operand with `extent` elements along its rows.  Copies past the
// extent are filled with zeros, so a short last chunk costs no memory traffic, and the MMAs that would only
// see zeros are left out.
static int pick_swizzle(long long extent) { return extent > 64 ? 128 : (extent > 32 ? 64 : 32); }
// Swizzle width of an MN-major operand of which a CTA stages `n` columns: the width that copies the fewest
// columns, the wider one of two equals.
static int pick_swizzle_mn(int n) {
  if (n <= 32) return 32;
  return (n + 127) / 128 * 128 <= (n + 63) / 64 * 64 ? 128 : 64;
}

struct MapSpec {
  int nd;
  cuuint64_t dims[4];
  cuuint64_t strides[3];   // bytes, dims 1..3
  cuuint32_t box[4];       // extent of the box in tensor elements (before the element stride)
  int swizzle;
  const void *base;
  cuuint32_t estr[4];      // element (traversal) stride per dimension; 0 = 1
  int im2col;              // 1: im2col map; box[0] = channels per pixel, box[1] = pixels per copy
  int lo[2], hi[2];        // its bounding box: first base pixel (W, H), last base pixel relative to the last pixel
};

static bool encode(niti_ctx *ctx, CUtensorMap *m, const MapSpec &s) {
  if (!ctx->encode_tiled) return false;
  if (((uintptr_t)s.base & 15) != 0) return false;
  for (int i = 0; i + 1 < s.nd; ++i)
    if (s.strides[i] % 16 != 0) return false;
  if (s.im2col) {
    if (!ctx->encode_im2col || s.box[1] > 256) return false;
    for (int i = 0; i < 2; ++i)
      if (s.lo[i] < -128 || s.lo[i] > 127 || s.hi[i] < -128 || s.hi[i] > 127) return false;
    const cuuint32_t es[4] = {1, s.estr[1] > 1 ? s.estr[1] : 1, s.estr[2] > 1 ? s.estr[2] : 1, 1};
    if (es[1] > 8 || es[2] > 8) return false;
    return ((EncodeIm2colFn)ctx->encode_im2col)(m, CU_TENSOR_MAP_DATA_TYPE_UINT8, 4, const_cast<void *>(s.base), s.dims,
                                                s.strides, s.lo, s.hi, s.box[0], s.box[1], es,
                                                CU_TENSOR_MAP_INTERLEAVE_NONE, swizzle_enum(s.swizzle),
                                                CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
                                                CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
  }
  for (int i = 0; i < s.nd; ++i)
    if (s.box[i] == 0 || s.box[i] > 256) return false;
  cuuint32_t es[4] = {1, 1, 1, 1};
  for (int i = 0; i < s.nd; ++i)
    if (s.estr[i] > 1) es[i] = s.estr[i];
  CUresult r = ((EncodeTiledFn)ctx->encode_tiled)(m, CU_TENSOR_MAP_DATA_TYPE_UINT8, (cuuint32_t)s.nd,
                                                  const_cast<void *>(s.base), s.dims, s.strides, s.box, es,
                                                  CU_TENSOR_MAP_INTERLEAVE_NONE, swizzle_enum(s.swizzle),
                                                  CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
                                                  CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS;
}

// Pixel box with Wt * Ht * Bt == 128 (powers of two).
static bool pick_pixel_box(int W, int H, int B, int &Wt, int &Ht, int &Bt) {
  Wt = 1;
  while (Wt < 128 && W % (Wt * 2) == 0) Wt *= 2;
  Ht = 1;
  while (Wt * Ht < 128 && H % (Ht * 2) == 0) Ht *= 2;
  Bt = 128 / (Wt * Ht);
  if (Bt > 256) return false;
  return Wt <= W && Ht <= H && Bt <= B;
}

// Tap groups of a weight gradient with few input channels.  With one tap per column tile every tap reads the error
// tensor again and a k-block's MMAs are shorter than its copies and barriers (about 400 cycles); a tile of several taps
// reads the error once for all of them.  The modelled cycles of all taps' k-blocks decide: MMAs (math or shared-memory
// reads), operand copies, or that floor.  Pairs of CTAs hold half of the taps each.  Measured, weight gradient with
// update: 5 x 5, 96 -> 256 channels, 27 x 27, batch 128 91.7 -> 60.5 us; 3 x 3, 24 -> 72, 64 x 64, batch 64 99.7 -> 60.6 us;
// 48 -> 96, 36 x 36, batch 100 37.9 -> 31.7 us; 32 -> 64, 28 x 28, batch 256 36.6 -> 26.6 us.
static int pick_tap_group(const GemmProblem &g, int ctas, int &cols) {
  cols = g.Ci <= 32 ? 32 : (g.Ci <= 64 ? 64 : 128);
  if (g.Ci > 128 || g.gk < 160 * 128) return 1;         // (few k-blocks: 96 -> 160 at 9 x 9, 64 k-blocks, 16.2 single, 17.9 grouped)
  const int taps = g.R * g.S;
  const double arows = g.Co / ctas < 128 ? (g.Co + ctas - 1) / ctas : 128;
  auto cost = [&](int t, int n) {
    const double mma = n / 2.0, smem = 32.0 + n / (4.0 * ctas);
    double c = 4.0 * (mma > smem ? mma : smem);
    const double copies = (arows + (double)n / ctas) * 128.0 / 84.0;
    if (c < copies) c = copies;
    if (c < 400.0) c = 400.0;
    return (double)((taps + t - 1) / t) * c;
  };
  int best_t = 1;
  double best = 0.95 * cost(1, (g.Ci + 31) / 32 * 32);
  for (int t = 2; t <= taps && t * cols <= 256; t += ctas)
    if (cost(t, t * cols) < best) { best = cost(t, t * cols); best_t = t; }
  return best_t;
}

constexpr size_t SMEM_BUDGET = 225 * 1024;            // dynamic shared memory beside the kernel's static arrays and alignment
constexpr size_t RED_BYTES = (size_t)EPI_WARPS * 4096;

// Map of the int32 accumulators for the reduce copies of a split contraction: 32 columns x 32 rows per copy, where
// the rows are consecutive rows, or one tap's rows of 32 output channels, or 32 pixels of a box.  Rows of a pitch
// that is no multiple of 16 bytes have no map (the epilogue then adds from registers).
static bool reduce_map(niti_ctx *ctx, const GemmProblem &g, TcParams &p, int32_t *acc, CUtensorMap &mc) {
  if (!ctx->encode_tiled || ((uintptr_t)acc & 15)) return false;
  const cuuint64_t row = (cuuint64_t)g.gn * 4;
  cuuint64_t dims[4] = {(cuuint64_t)g.gn, (cuuint64_t)g.gm, 1, 1};
  cuuint64_t strides[3] = {row, row * (cuuint64_t)g.gm, row * (cuuint64_t)g.gm};
  cuuint32_t box[4] = {32, 32, 1, 1};
  const cuuint32_t es[4] = {1, 1, 1, 1};
  int red = 1;
  if (g.kind == GK_CONV_WGRAD) {
    dims[0] = (cuuint64_t)p.Cn; dims[1] = (cuuint64_t)g.R * g.S; dims[2] = (cuuint64_t)g.Co;
    strides[0] = (cuuint64_t)p.Cn * 4; strides[1] = row; strides[2] = row * (cuuint64_t)g.Co;
    box[1] = 1; box[2] = 32;
  } else if ((g.kind == GK_CONV_FWD || g.kind == GK_CONV_DGRAD) && !p.i2c) {
    red = 2;
    dims[1] = (cuuint64_t)p.PW; dims[2] = (cuuint64_t)p.PH; dims[3] = (cuuint64_t)p.PB;
    strides[1] = row * p.PW; strides[2] = row * p.PW * p.PH;
    box[1] = p.Wt < 32 ? p.Wt : 32;
    box[2] = p.Ht < 32 / (int)box[1] ? p.Ht : 32 / box[1];
    box[3] = 32 / (box[1] * box[2]);
  }
  if ((strides[0] & 15) || (strides[1] & 15) || strides[2] >= (1ull << 40)) return false;
  if (((EncodeTiledFn)ctx->encode_tiled)(&mc, CU_TENSOR_MAP_DATA_TYPE_INT32, 4, acc, dims, strides, box, es,
                                         CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                                         CU_TENSOR_MAP_L2_PROMOTION_NONE, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
    return false;
  p.red = red;
  return true;
}

// Extents and strides of a tensor of overlapping windows (see WindowGeometry at the boundary): a window's channels,
// the windows of a row, rows, images.
static void window_map(const GemmProblem &g, MapSpec &s) {
  s.dims[0] = (cuuint64_t)g.win_chans;
  s.strides[0] = (cuuint64_t)g.win_sw;
  s.strides[1] = (cuuint64_t)g.win_sh;
  s.strides[2] = (cuuint64_t)g.win_sh * g.H;
}

// The patches of the resident-weights mode cover 8 x 16 pixels: images that fill at least
// three quarters of them, or are large enough.
static bool halo_fits(int W, int H) {
  const int cover = (W + 7) / 8 * 8 * ((H + 15) / 16 * 16);
  return (W >= 10 && H >= 18) || 4 * W * H >= 3 * cover;
}

static int round_up32(long long n) { return (int)((n + 31) / 32 * 32); }

// Width of a column tile: the fewest tiles of at most 256 columns, all of about the same width.
static int pick_bn(long long gn) {
  const long long tiles = (gn + 255) / 256;
  return round_up32((gn + tiles - 1) / tiles);
}

// Contractions up to this length run on single CTAs, deeper ones on CTA pairs (see niti_tc_gemm's choice of a plan).
constexpr long long PAIR_MIN_K = 1152;

// The same for an operand that is staged with its columns contiguous (errors and weight gradients): chunks of at least 64
// columns, because 96 are staged as 32-byte rows.  Wide swizzles pay in deep contractions, where the operand copies and the
// shared-memory reads are the bound (error of a 5 x 5 layer with 96 input channels 81.8 -> 71.8 us, weight gradient with
// 160 channels at 28 x 28 33.4 -> 29.7 us); in short ones the wider accumulator only costs the epilogue (16.6 -> 17.7 us).
static int pick_bn_mn(long long gn, long long gk) {
  const int w = pick_bn(gn);
  return w > 64 && gk > PAIR_MIN_K ? (w + 63) / 64 * 64 : w;
}

// Builds params and maps; returns false if the shape is not eligible for this engine.
// `aligned`: output (and mask) pointers and rows are 32-byte aligned.
// force_bn: column tile of an unsplit one-wave plan (see pick_one_wave), 0 for the planner's own choice, -1 for that
// without tap groups.
// want: ANY, or only a plan in the resident-weights / tap-pair mode (HALO) or the row-batched mode (BATCHED).
enum PlanWant { PLAN_ANY = 0, PLAN_HALO = 1, PLAN_BATCHED = 2 };
static bool plan(niti_ctx *ctx, const GemmProblem &g, int ctas, PlanWant want, bool aligned, int force_bn, int32_t *acc, TcParams &p, CUtensorMap &ma,
                 CUtensorMap &mb, CUtensorMap &mc) {
  memset(&p, 0, sizeof(p));
  p.ctas = ctas;
  p.kind = g.kind;
  p.gm = g.gm;
  p.gn = g.gn;
  p.splits = 1;
  p.mode = aligned ? 0 : 1;
  MapSpec sa, sb;
  memset(&sa, 0, sizeof(sa));
  memset(&sb, 0, sizeof(sb));
  int a_mn = 0, b_mn = 0;        // 1 = MN-major operand
  int a_sw = 0, b_sw = 0;
  int tail = 0;                  // contraction elements of the last chunk of c_chunks when it is not a whole one
  long long m_tiles = 0;
  // (rows, columns and contraction elements are counted in 32 bits, and divided by div_by)
  if (g.gm * g.gn >= (1LL << 31) || g.gm >= (1LL << 31) - 1024 || g.gk >= (1LL << 31) - 1024) return false;
  // operands as they are copied: padded where the caller's rows are no multiple of 16 bytes
  const int8_t *q0 = g.q0 ? g.q0 : g.p0, *q1 = g.q1 ? g.q1 : g.p1;
  if (g.kind == GK_FC_DGRAD && g.gk < 32) return false;            // (10-class heads: the CUDA-core engine is faster)
  if (g.kind == GK_FC_WGRAD && (g.gm < 32 || g.gk < 32)) return false;
  switch (g.kind) {
    case GK_FC_FWD: {
      p.kdepth = pick_swizzle(g.gk);
      p.bn = force_bn > 0 ? force_bn : pick_bn(g.gn);
      a_sw = b_sw = p.kdepth;
      const cuuint64_t ld0 = (cuuint64_t)(g.ld0 ? g.ld0 : g.gk), ld1 = (cuuint64_t)(g.ld1 ? g.ld1 : g.gk);
      sa = {2, {(cuuint64_t)g.gk, (cuuint64_t)g.gm}, {ld0}, {(cuuint32_t)p.kdepth, BM}, a_sw, q0};
      sb = {2, {(cuuint64_t)g.gk, (cuuint64_t)g.gn}, {ld1}, {(cuuint32_t)p.kdepth, (cuuint32_t)(p.bn / ctas)}, b_sw, q1};
      p.kb_total = (int)((g.gk + p.kdepth - 1) / p.kdepth);
      m_tiles = (g.gm + BM - 1) / BM;
      p.n_tiles_n = (int)((g.gn + p.bn - 1) / p.bn);
      break;
    }
    case GK_FC_DGRAD: {   // out [M][K'], contraction over N
      p.kdepth = pick_swizzle(g.gk);
      b_mn = 1;
      p.bn = force_bn > 0 ? force_bn : pick_bn_mn(g.gn, g.gk);
      b_sw = pick_swizzle_mn(p.bn / ctas);
      a_sw = p.kdepth;
      const cuuint64_t ld0 = (cuuint64_t)(g.ld0 ? g.ld0 : g.gk), ld1 = (cuuint64_t)(g.ld1 ? g.ld1 : g.gn);
      sa = {2, {(cuuint64_t)g.gk, (cuuint64_t)g.gm}, {ld0}, {(cuuint32_t)p.kdepth, BM}, a_sw, q0};
      sb = {2, {(cuuint64_t)g.gn, (cuuint64_t)g.gk}, {ld1}, {(cuuint32_t)b_sw, (cuuint32_t)p.kdepth}, b_sw, q1};
      p.kb_total = (int)((g.gk + p.kdepth - 1) / p.kdepth);
      m_tiles = (g.gm + BM - 1) / BM;
      p.n_tiles_n = (int)((g.gn + p.bn - 1) / p.bn);
      break;
    }
    case GK_FC_WGRAD: {   // out [N][K'], contraction over M (rows of both operands)
      a_mn = b_mn = 1;
      a_sw = pick_swizzle(g.gm);
      p.kdepth = pick_swizzle(g.gk);
      p.bn = force_bn > 0 ? force_bn : pick_bn_mn(g.gn, g.gk);
      b_sw = pick_swizzle_mn(p.bn / ctas);
      const cuuint64_t ld0 = (cuuint64_t)(g.ld0 ? g.ld0 : g.gm), ld1 = (cuuint64_t)(g.ld1 ? g.ld1 : g.gn);
      sa = {2, {(cuuint64_t)g.gm, (cuuint64_t)g.gk}, {ld0}, {(cuuint32_t)a_sw, (cuuint32_t)p.kdepth}, a_sw, q0};
      sb = {2, {(cuuint64_t)g.gn, (cuuint64_t)g.gk}, {ld1}, {(cuuint32_t)b_sw, (cuuint32_t)p.kdepth}, b_sw, q1};
      p.kb_total = (int)((g.gk + p.kdepth - 1) / p.kdepth);
      m_tiles = (g.gm + BM - 1) / BM;
      p.n_tiles_n = (int)((g.gn + p.bn - 1) / p.bn);
      break;
    }
    case GK_CONV_FWD:
    case GK_CONV_DGRAD: {
      // Rows run over the pixels of the OUTPUT tensor of this multiply (forward: the Ho x Wo output;
      // error: the H x W input-shaped tensor); the shifted operand is the other activation tensor and
      // may have another size (padding other than (R-1)/2, strides): its copies start at any
      // coordinate and read zeros outside it.  A forward stride becomes the element stride of those
      // copies; the error of a strided convolution runs over the phases of its input grid (see dstride).
      const bool fwd = g.kind == GK_CONV_FWD;
      const int st = g.stride > 1 ? g.stride : 1;
      const int RW = fwd ? g.Wo : g.W, RH = fwd ? g.Ho : g.H;      // pixel grid of the rows
      const int OW = fwd ? g.W : g.Wo, OH = fwd ? g.H : g.Ho;      // pixel grid of the shifted operand
      const bool same = g.Ho == g.H && g.Wo == g.W && st == 1;
      const int Cc = fwd ? g.Ci : g.Co;        // contraction channels
      const int Cn = fwd ? g.Co : g.Ci;        // output channels of this multiply
      const long long ld0 = g.ld0 ? g.ld0 : Cc, ld1 = g.ld1 ? g.ld1 : g.Ci;       // pixel pitch, tap pitch of w
      p.kdepth = pick_swizzle(Cc);
      tail = Cc % p.kdepth;
      const int pad_w = g.win_chans ? 0 : g.pad;
      p.R = g.R; p.S = g.S; p.pad = g.pad;
      p.stride = fwd ? st : 1;
      p.stride_w = g.win_chans ? 1 : p.stride;
      p.dstride = fwd ? 1 : st;
      p.c_chunks = (Cc + p.kdepth - 1) / p.kdepth;
      p.Cn = Cn;
      a_sw = p.kdepth;
      // Pixel rows.  Where a pixel box of 128 tiles the image exactly (and no stride is involved) a tile of output
      // rows is such a box: it allows the fused 2 x 2 pooling.  Everywhere else (odd image sides, strides) the
      // rows of a tile are 128 consecutive pixels of the flattened grid, copied in im2col mode, which walks the
      // grid pixel by pixel, image after image, with the convolution's stride and zero padding.
      p.i2c = (st > 1 || g.win_chans || !pick_pixel_box(RW, RH, g.B, p.Wt, p.Ht, p.Bt)) ? 1 : 0;
      sa = {4, {(cuuint64_t)Cc, (cuuint64_t)OW, (cuuint64_t)OH, (cuuint64_t)g.B},
            {(cuuint64_t)ld0, (cuuint64_t)ld0 * OW, (cuuint64_t)ld0 * OW * OH},
            {(cuuint32_t)p.kdepth, (cuuint32_t)p.Wt, (cuuint32_t)p.Ht, (cuuint32_t)p.Bt}, a_sw, q0};
      if (g.win_chans) window_map(g, sa);
      p.PW = RW; p.PH = RH; p.PB = g.B;
      p.T_r = g.R; p.T_s = g.S;
      if (p.i2c) {
        if (g.R > 256 || g.S > 256) return false;
        p.Wt = p.Ht = p.Bt = 1;
        sa.im2col = 1;
        sa.box[1] = BM;
        if (fwd) {
          p.i2c_w0 = -pad_w; p.i2c_h0 = -g.pad;
          sa.estr[1] = (cuuint32_t)p.stride_w; sa.estr[2] = (cuuint32_t)st;
          sa.hi[0] = pad_w - (g.S - 1); sa.hi[1] = g.pad - (g.R - 1);
        } else {
          // phases of the input grid (a single one without a stride): grid position u of phase f is input row
          // st * (u + u0) + f - pad and collects e[u + u0 - t] for the taps f + st * t.  All phases share the grid
          // of the widest one; positions outside the tensor are masked.
          p.nph_r = st < g.R ? st : g.R; p.nph_s = st < g.S ? st : g.S;
          p.T_r = (g.R + st - 1) / st; p.T_s = (g.S + st - 1) / st;
          const int fr = g.pad - (p.nph_r - 1), fs = g.pad - (p.nph_s - 1);
          p.u0_r = fr > 0 ? (fr + st - 1) / st : 0; p.u0_s = fs > 0 ? (fs + st - 1) / st : 0;
          const int u1_r = (g.H - 1 + g.pad) / st, u1_s = (g.W - 1 + g.pad) / st;
          p.PH = u1_r - p.u0_r + 1; p.PW = u1_s - p.u0_s + 1;
          if (p.PH <= 0 || p.PW <= 0) return false;      // (every window row or column lies in the padding: all errors are 0)
          p.i2c_h0 = p.u0_r - (p.T_r - 1); p.i2c_w0 = p.u0_s - (p.T_s - 1);
          sa.hi[0] = p.i2c_w0 + p.PW - 1 - (OW - 1); sa.hi[1] = p.i2c_h0 + p.PH - 1 - (OH - 1);
          p.OH = g.H; p.OW = g.W;
        }
        sa.lo[0] = p.i2c_w0; sa.lo[1] = p.i2c_h0;
        if ((long long)p.PB * p.PH * p.PW >= (1LL << 31) - 512) return false;
      }
      p.w_tiles = (p.PW + p.Wt - 1) / p.Wt;
      p.h_tiles = (p.PH + p.Ht - 1) / p.Ht;
      p.b_tiles = (g.B + p.Bt - 1) / p.Bt;
      m_tiles = (long long)p.w_tiles * p.h_tiles * p.b_tiles;
      if (p.i2c) m_tiles = (m_tiles + BM - 1) / BM;
      p.bn = force_bn > 0 ? force_bn : fwd ? pick_bn(Cn) : pick_bn_mn(Cn, g.gk);
      if (fwd && ctas == 2 && Cn > 256 && force_bn <= 0) {
        // Whole waves: with 256-wide tiles the 14 x 14 layers are 98 tile pairs on 74 pairs of SMs, two
        // waves of which the second is a third full; 192-wide tiles make 147 items, two full waves.
        // (A 192-wide MMA takes as long as a 256-wide one, so an item is not shorter; it moves three
        // quarters of the weights.  Measured 31.0 against 31.5 us; 128-wide tiles, three waves of
        // half the math each, are bound by the shared-memory traffic of their operands: 38.4 us.)
        const long long mu = (m_tiles + 1) / 2, units = ctx->sm_count / 2;
        const long long w256 = (mu * ((Cn + 255) / 256) + units - 1) / units;
        const long long w192 = (mu * ((Cn + 191) / 192) + units - 1) / units;
        if (w192 * 192 * 10 < w256 * 256 * 9) p.bn = 192;
      }
      if (p.i2c || tail || g.q0 || g.q1 || g.Ci % 32 != 0) p.mode = 1;
      // (a copy of w may reach into the next tap's columns only where those are not multiplied)
      if (!fwd && Cn % pick_swizzle_mn(p.bn / ctas) != 0) p.mode = 1;
      if (p.dstride > 1) p.mode = 2;
      // w viewed as [Co][R*S][Ci]
      sb = {3, {(cuuint64_t)g.Ci, (cuuint64_t)g.R * g.S, (cuuint64_t)g.Co},
            {(cuuint64_t)ld1, (cuuint64_t)ld1 * g.R * g.S}, {(cuuint32_t)p.kdepth, 1, (cuuint32_t)(p.bn / ctas)}, p.kdepth, q1};
      if (!fwd) {
        b_mn = 1;
        sb.swizzle = pick_swizzle_mn(p.bn / ctas);
        sb.box[0] = (cuuint32_t)sb.swizzle;
        sb.box[2] = (cuuint32_t)p.kdepth;
      }
      b_sw = sb.swizzle;
      if (p.mode == 0) {       // (plain matrices: [Cn][R*S*Ci], and [Co][R*S*Ci] with column tap * Ci + ci)
        const cuuint64_t row = (cuuint64_t)g.R * g.S * g.Ci;
        sb.nd = 2;
        sb.dims[0] = row; sb.dims[1] = (cuuint64_t)g.Co;
        sb.strides[0] = row;
        sb.box[1] = sb.box[2];
      }
      p.kb_total = g.R * g.S * p.c_chunks;
      p.n_tiles_n = (Cn + p.bn - 1) / p.bn;
      if (p.dstride > 1) p.kb_total = p.T_r * p.T_s * p.c_chunks;                 // (of the longest phase)
      // halo mode: one channel chunk, one column tile, weights of all taps fit beside >= 3 patches
      // (short channel chunks and padded operands need the general instance, whose weights come through a 3-D map)
      if (want == PLAN_HALO && same && ctas == 1 && g.R == 3 && g.S == 3 && g.pad == 1 && p.c_chunks == 1 &&
          p.n_tiles_n == 1 && halo_fits(g.W, g.H) && Cn % 8 == 0) {
        const int a_stage = (180 * p.kdepth + 1023) / 1024 * 1024;
        const int tap_cols = fwd ? p.bn : (p.bn + b_sw - 1) / b_sw * b_sw;        // (columns past Cn are not multiplied)
        const int b_res = (9 * tap_cols * p.kdepth + 1023) / 1024 * 1024;
        if (b_res + 3 * a_stage <= 224 * 1024) {
          p.halo = 1;
          p.i2c = 0;
          p.mode = aligned && !tail && !g.q0 && !g.q1 && (fwd || Cn % 32 == 0) ? 0 : 1;
          sa.im2col = 0;
          p.PW = g.W; p.PH = g.H;
          p.Wt = 8; p.Ht = 16; p.Bt = 1;
          p.w_tiles = (g.W + 7) / 8;
          p.h_tiles = (g.H + 15) / 16;
          p.b_tiles = g.B;
          m_tiles = (long long)p.w_tiles * p.h_tiles * p.b_tiles;
          sa.box[1] = 10; sa.box[2] = 18; sa.box[3] = 1;
          if (p.mode == 1) {
            sb = {3, {(cuuint64_t)g.Ci, 9, (cuuint64_t)g.Co}, {(cuuint64_t)ld1, (cuuint64_t)9 * ld1},
                  {(cuuint32_t)b_sw, 1, (cuuint32_t)(fwd ? p.bn : p.kdepth)}, b_sw, q1};
          } else if (fwd) {
            sb = {2, {(cuuint64_t)g.gk, (cuuint64_t)Cn}, {(cuuint64_t)g.gk}, {(cuuint32_t)p.kdepth, (cuuint32_t)p.bn}, b_sw, q1};
          } else {       // w viewed as [Co rows][9 * Ci]: column = tap * Ci + ci
            sb = {2, {(cuuint64_t)9 * g.Ci, (cuuint64_t)g.Co}, {(cuuint64_t)9 * g.Ci}, {(cuuint32_t)b_sw, (cuuint32_t)p.kdepth}, b_sw, q1};
          }
          p.b_tile_bytes = tap_cols * p.kdepth;
          p.b_res_bytes = b_res;
        }
      }
      break;
    }
    case GK_CONV_WGRAD: {
      // the contraction runs over the pixels of the OUTPUT grid (Ho x Wo); the input tensor is copied
      // shifted by the tap, with the stride as element stride
      const int st = g.stride > 1 ? g.stride : 1;
      const bool same = g.Ho == g.H && g.Wo == g.W && st == 1;
      p.stride = st;
      // (64 x 64)-channel blocks re-read the activations once per block of the other operand and their N = 64 MMAs run
      // at two thirds of the rate: this mode is kept where the tap groups below would leave half of the MMA's rows
      // empty (64 output channels, batch 64: this / groups 121 / 211 us at 224 x 224, 40 / 66 at 112 x 112, 21 / 23 at 56 x
      // 56, 14.4 / 14.8 at 28 x 28; 128 input channels 65 / 113 and 29 / 38, 192 91 / 156, 256 47 / 62) or spend as much on
      // copies (128 -> 128: 115 / 125 at 112 x 112, 43 / 43 at 56 x 56, 22 / 21 at 28 x 28).  Elsewhere the groups are as
      // good or better: 64 -> 128 65 / 65, 28 / 24 and 17 / 16 us, 64 -> 192 35 / 38, 64 -> 256 41 / 39, 128 -> 256 75 / 59
      if (want == PLAN_HALO && same && ctas == 1 && g.R == 3 && g.S == 3 && g.pad == 1 && g.Ci % 64 == 0 && g.Co % 64 == 0 &&
          g.W >= 10 && g.H >= 18 && (long long)g.Ci * g.Co <= 16384 && (g.Co == 64 || g.Ci >= 128) && !g.q0 && !g.q1) {
        p.halo = 2;
        p.kdepth = 128;
        p.bn = 64;
        p.Wt = 8; p.Ht = 16; p.Bt = 1;
        p.w_tiles = (g.W + 7) / 8;
        p.h_tiles = (g.H + 15) / 16;
        p.b_tiles = g.B;
        p.PW = g.W; p.PH = g.H; p.PB = g.B;
        p.Cn = g.Ci;
        p.wg_nci = g.Ci / 64;
        p.kb_total = p.w_tiles * p.h_tiles * p.b_tiles;      // pixel tiles
        // A = input patch (p1 = x), B = error tile (p0 = e); both MN-major, 64-byte rows
        sa = {4, {(cuuint64_t)g.Ci, (cuuint64_t)g.W, (cuuint64_t)g.H, (cuuint64_t)g.B},
              {(cuuint64_t)g.Ci, (cuuint64_t)g.Ci * g.W, (cuuint64_t)g.Ci * g.W * g.H}, {64, 10, 18, 1}, 64, g.p1};
        sb = {4, {(cuuint64_t)g.Co, (cuuint64_t)g.W, (cuuint64_t)g.H, (cuuint64_t)g.B},
              {(cuuint64_t)g.Co, (cuuint64_t)g.Co * g.W, (cuuint64_t)g.Co * g.W * g.H}, {64, 8, 16, 1}, 64, g.p0};
        p.a_box_bytes = 180 * 64; p.b_box_bytes = 128 * 64;
        p.a_bytes = 12288; p.b_bytes = 8192;
        p.a_boxes = p.b_boxes = 1;
        p.stages = MAX_STAGES;
        p.nprod = 2;                                          // divides the eight stages
        p.nbuf = 5;                                           // five accumulators of 64 columns
        p.ksteps = 4;
        // MN-major, 64-byte swizzle: 8-row groups one patch row (10 pixels) apart for A, contiguous for B;
        // the leading-dimension field of A is filled per tap pair by the kernel
        p.a_desc = ((unsigned long long)((10 * 64) >> 4) << 32) | ((unsigned long long)1 << 46) | layout_bits(64);
        p.b_desc = ((unsigned long long)1 << 16) | ((unsigned long long)((8 * 64) >> 4) << 32) |
                   ((unsigned long long)1 << 46) | layout_bits(64);
        p.idesc = (2u << 4) | (1u << 7) | (1u << 10) | (1u << 15) | (1u << 16) | ((unsigned)(64 >> 3) << 17) |
                  ((unsigned)(BM >> 4) << 24);
        const long long blocks = (long long)(g.Ci / 64) * (g.Co / 64);
        // split the pixel range so that the items fill whole waves of SMs
        int best_s = 1;
        double best_eff = 0;
        const int max_s = p.kb_total / 4 > 0 ? p.kb_total / 4 : 1;
        for (int sp = 1; sp <= max_s && sp <= 4 * ctx->sm_count && best_eff < 0.98; ++sp) {
          const int it = (int)blocks * sp;
          const int waves = (it + ctx->sm_count - 1) / ctx->sm_count;
          const double eff = (double)it / (double)(waves * ctx->sm_count);
          if (eff > best_eff + 0.02) { best_eff = eff; best_s = sp; }
        }
        p.splits = best_s;
        // (a split covers at most NITI_SPLIT_MAX_K pixels: its partial sums cannot wrap)
        if (p.splits < (p.kb_total + NITI_SPLIT_MAX_K / 128 - 1) / (NITI_SPLIT_MAX_K / 128))
          p.splits = (p.kb_total + NITI_SPLIT_MAX_K / 128 - 1) / (NITI_SPLIT_MAX_K / 128);
        if (p.splits > NITI_MAX_SPLITS) return false;
        p.kb_per_split = (p.kb_total + p.splits - 1) / p.splits;
        p.splits = (p.kb_total + p.kb_per_split - 1) / p.kb_per_split;
        p.items = blocks * p.splits;
        p.m_units = 1;
        p.n_tiles_n = 1;
        if (!reduce_map(ctx, g, p, acc, mc)) return false;
        p.red_off = p.stages * (p.a_bytes + p.b_bytes);
        if (!encode(ctx, &ma, sa) || !encode(ctx, &mb, sb)) return false;
        return true;
      }
      if (want == PLAN_HALO) return false;
      a_mn = b_mn = 1;
      const long long ld0 = g.ld0 ? g.ld0 : g.Co, ld1 = g.ld1 ? g.ld1 : g.Ci;     // pixel pitches of e and x
      a_sw = pick_swizzle(g.Co);
      p.kdepth = 128;
      p.PW = g.Wo; p.PH = g.Ho; p.PB = g.B;
      p.R = g.R; p.S = g.S; p.pad = g.pad;
      p.Cn = g.Ci;
      p.bn = force_bn > 0 ? force_bn : pick_bn_mn(g.Ci, g.gk);
      b_sw = pick_swizzle_mn(p.bn / ctas);
      p.n_chunks = (g.Ci + p.bn - 1) / p.bn;
      p.tg = 1;
      if (force_bn == 0) {
        const int t = pick_tap_group(g, ctas, p.tg_cols);
        if (t > 1) {
          p.tg = t;
          p.bn = t * p.tg_cols;
          p.n_chunks = 1;
          b_sw = p.tg_cols;                       // (32, 64 or 128: one copy per tap)
        }
      }
      // (pixel boxes or runs of consecutive pixels: see "Pixel rows" above; a run of e is a piece of a matrix)
      p.stride_w = g.win_chans ? 1 : st;
      p.i2c = (st > 1 || g.win_chans || !pick_pixel_box(g.Wo, g.Ho, g.B, p.Wt, p.Ht, p.Bt)) ? 1 : 0;
      if (p.i2c) p.mode = 1;
      sb = {4, {(cuuint64_t)g.Ci, (cuuint64_t)g.W, (cuuint64_t)g.H, (cuuint64_t)g.B},
            {(cuuint64_t)ld1, (cuuint64_t)ld1 * g.W, (cuuint64_t)ld1 * g.W * g.H},
            {(cuuint32_t)b_sw, (cuuint32_t)p.Wt, (cuuint32_t)p.Ht, (cuuint32_t)p.Bt}, b_sw, q1};
      if (g.win_chans) window_map(g, sb);
      if (p.i2c) {
        if (g.R > 256 || g.S > 256) return false;
        p.Wt = p.Ht = p.Bt = 1;
        const int pad_w = g.win_chans ? 0 : g.pad;
        p.i2c_w0 = -pad_w; p.i2c_h0 = -g.pad;
        p.i2c_dj = BM % g.Wo;
        p.i2c_di = BM / g.Wo % g.Ho;
        p.i2c_db = BM / g.Wo / g.Ho;
        sa = {2, {(cuuint64_t)g.Co, (cuuint64_t)g.gk}, {(cuuint64_t)ld0}, {(cuuint32_t)a_sw, (cuuint32_t)p.kdepth}, a_sw, q0};
        sb.im2col = 1;
        sb.box[1] = (cuuint32_t)p.kdepth;
        sb.estr[1] = (cuuint32_t)p.stride_w; sb.estr[2] = (cuuint32_t)st;
        sb.lo[0] = -pad_w; sb.lo[1] = -g.pad;
        sb.hi[0] = pad_w - (g.S - 1); sb.hi[1] = g.pad - (g.R - 1);
        if (g.gk >= (1LL << 31) - 512) return false;
      } else {
        sa = {4, {(cuuint64_t)g.Co, (cuuint64_t)g.Wo, (cuuint64_t)g.Ho, (cuuint64_t)g.B},
              {(cuuint64_t)ld0, (cuuint64_t)ld0 * g.Wo, (cuuint64_t)ld0 * g.Wo * g.Ho},
              {(cuuint32_t)a_sw, (cuuint32_t)p.Wt, (cuuint32_t)p.Ht, (cuuint32_t)p.Bt}, a_sw, q0};
      }
      p.w_tiles = (g.Wo + p.Wt - 1) / p.Wt;
      p.h_tiles = (g.Ho + p.Ht - 1) / p.Ht;
      p.b_tiles = (g.B + p.Bt - 1) / p.Bt;
      p.kb_total = p.w_tiles * p.h_tiles * p.b_tiles;
      if (p.i2c) p.kb_total = (int)((g.gk + p.kdepth - 1) / p.kdepth);
      m_tiles = (g.Co + BM - 1) / BM;
      p.n_tiles_n = (g.R * g.S + p.tg - 1) / p.tg * p.n_chunks;
      break;
    }
    default:
      return false;
  }
  if (want == PLAN_HALO && !p.halo) return false;
  p.ksteps = p.kdepth / 32;
  if (tail && (tail + 31) / 32 < p.ksteps) {
    p.tail_ks = (tail + 31) / 32;
    if (p.c_chunks == 1) { p.ksteps = p.tail_ks; p.tail_ks = 0; }                // every chunk is the short one
  }
  // operand staging
  if (a_mn) {
    p.a_boxes = BM / a_sw;
    if ((long long)p.a_boxes * a_sw > (g.gm + a_sw - 1) / a_sw * a_sw) p.a_boxes = (int)((g.gm + a_sw - 1) / a_sw);
    p.a_box_bytes = p.kdepth * a_sw;
    p.a_box_step = a_sw;
    p.a_bytes = (BM / a_sw) * p.a_box_bytes;
    p.a_desc = desc_mnmajor(a_sw, p.kdepth);
    p.a_kstep16 = (unsigned)((32 * a_sw) >> 4);
  } else {
    p.a_boxes = 1;
    p.a_box_bytes = BM * p.kdepth;
    p.a_bytes = p.a_box_bytes;
    p.a_desc = desc_kmajor(a_sw);
    p.a_kstep16 = 2;
  }
  // Row-batched mode: a multiply with one or two k-blocks and a narrow output (the gathered first
  // layer: K = 32, N = 64) is all per-tile bookkeeping.  One item then covers mrep 128-row tiles: one
  // stage holds their A boxes, one MMA per tile writes its own bn_mma columns of the accumulator,
  // and the barriers, commits and tile decoding are paid once per item.
  p.mrep = 1;
  if (g.kind == GK_FC_FWD && ctas == 1 && ctx->engine != 4 && !g.in_place && p.n_tiles_n == 1 && p.kb_total <= 2 && p.bn <= 128 &&
      m_tiles >= 8LL * ctx->sm_count) {
    p.mrep = p.bn <= 64 ? 4 : 2;
    p.a_boxes = p.mrep;
    p.a_bytes = p.mrep * p.a_box_bytes;
    m_tiles = (m_tiles + p.mrep - 1) / p.mrep;
  }
  if (want == PLAN_BATCHED && p.mrep == 1) return false;
  const int bn_cta = p.bn / ctas;               // output columns staged by each CTA
  if (bn_cta % 16) return false;
  if (b_mn) {
    p.b_boxes = (bn_cta + b_sw - 1) / b_sw;
    p.tg_boxes = p.tg > 1 ? 1 : p.b_boxes;
    p.b_box_bytes = p.kdepth * b_sw;
    p.b_box_step = b_sw;
    p.b_bytes = p.b_boxes * p.b_box_bytes;
    p.b_desc = desc_mnmajor(b_sw, p.kdepth);
    p.b_kstep16 = (unsigned)((32 * b_sw) >> 4);
  } else {
    p.b_boxes = 1;
    p.b_box_bytes = bn_cta * p.kdepth;
    p.b_bytes = p.b_box_bytes;
    p.b_desc = desc_kmajor(b_sw);
    p.b_kstep16 = 2;
  }
  // stage buffers must start on the swizzle period (1024 bytes)
  p.a_bytes = (p.a_bytes + 1023) / 1024 * 1024;
  p.b_bytes = (p.b_bytes + 1023) / 1024 * 1024;
  int stage_bytes = p.a_bytes + p.b_bytes;
  p.stages = (200 * 1024) / stage_bytes;
  if (p.halo) {
    // a stage is one 10 x 18 pixel patch; consecutive 8-row groups of a tap are one patch row apart
    p.a_box_bytes = 180 * p.kdepth;
    p.a_bytes = (p.a_box_bytes + 1023) / 1024 * 1024;
    p.a_desc = desc_kmajor(a_sw, 10);
    p.b_bytes = 0;
    stage_bytes = p.a_bytes;
    p.stages = (224 * 1024 - p.b_res_bytes) / stage_bytes;
  }
  if (p.stages > MAX_STAGES) p.stages = MAX_STAGES;
  if (p.stages < 2) return false;
  // instruction descriptor: s32 accumulate, signed 8-bit operands, majorness, N, M
  p.idesc = (2u << 4) | (1u << 7) | (1u << 10) | ((unsigned)a_mn << 15) | ((unsigned)b_mn << 16) |
            ((unsigned)(p.bn >> 3) << 17) | ((unsigned)((BM * ctas) >> 4) << 24);
  p.bn_mma = p.bn;
  p.bn *= p.mrep;
  p.m_units = (int)((m_tiles + ctas - 1) / ctas);
  long long tiles = (long long)p.m_units * p.n_tiles_n;
  const int units = ctx->sm_count / ctas;       // CTAs (or CTA pairs) that run at the same time
  // visit row units in groups so that concurrently running tiles share operands in L2
  if ((g.kind == GK_FC_FWD || g.kind == GK_FC_DGRAD || g.kind == GK_FC_WGRAD) && p.n_tiles_n > 1 && p.m_units > 1)
    p.raster_g = ctas == 2 ? 8 : 12;
  // split the contraction when the tiles alone cannot fill the SMs
  if (tiles < units && p.kb_total >= 8 && p.dstride <= 1 && force_bn <= 0) {
    // pick the split count with the least modelled time: waves of items, each item running its
    // share of the k-blocks plus a fixed cost (pipeline fill and the epilogue's reduce copies) of about
    // four k-blocks
    double best = 1e30;
    int best_s = 1;
    int max_s = p.kb_total / 4;
    for (int sp = 1; sp <= max_s && sp <= 4 * units; ++sp) {
      const int it = (int)tiles * sp;
      const int waves = (it + units - 1) / units;
      // (no later split count can cost less than this: the host time of the search counts in short calls)
      if ((double)tiles * p.kb_total / units + 4.0 * waves >= best * 0.98) break;
      const double cost = (double)waves * ((double)((p.kb_total + sp - 1) / sp) + 4.0);
      if (cost < best * 0.98) { best = cost; best_s = sp; }
    }
    p.splits = best_s;
  }
  {
    // a contraction longer than NITI_SPLIT_MAX_K is always split, into pieces whose partial sums cannot
    // wrap an int32; the epilogue records the largest partial sum of every piece (overflow detection)
    const int max_kb = NITI_SPLIT_MAX_K / p.kdepth;
    const int min_splits = (p.kb_total + max_kb - 1) / max_kb;
    if (p.splits < min_splits) p.splits = min_splits;
    if (force_bn > 0 && p.splits > 1) return false;
    if (p.splits > NITI_MAX_SPLITS || (p.splits > 1 && p.dstride > 1)) return false;
  }
  p.kb_per_split = (p.kb_total + p.splits - 1) / p.splits;
  p.splits = (p.kb_total + p.kb_per_split - 1) / p.kb_per_split;
  if (p.splits > 1 && !p.halo && reduce_map(ctx, g, p, acc, mc)) {
    int st = (int)(SMEM_BUDGET - RED_BYTES) / stage_bytes;
    if (st > MAX_STAGES) st = MAX_STAGES;
    if (st >= 2) {
      p.stages = st;
      p.red_off = st * stage_bytes;
    } else {
      p.red = 0;
    }
  }
  // (tap groups only where the sums leave through reduce copies, which place every tap's columns)
  if (p.tg > 1 && !(p.splits > 1 && p.red)) return plan(ctx, g, ctas, want, aligned, -1, acc, p, ma, mb, mc);
  // All of B resident: with one column tile every tile reads the same B tiles again, and short contractions are bound by their
  // copies (about 4 cycles a row).  Where they leave room for the A stages, the first tile of a CTA copies them and the others
  // find them.  Before -> after: 11 x 11 stride 4 RGB 61.7 -> 49.8 us, 5 x 5 RGB at 64 x 64 to 64 and 96 channels 45.0 -> 30.1
  // and 51.2 -> 34.9, 1 x 1 64 -> 256 at 56 x 56 28.6 -> 27.3, error of 1 x 1 48 -> 384 at 45 x 45 27.8 -> 18.5, 72 -> 40 at 32 x
  // 32 19.0 -> 17.3; row-batched, at any row width, 3 x 3 RGB at 112 x 112 47.4 -> 44.1, 200000 x 32 x 27 18.8 -> 17.8, x 64 x 64
  // 16.0 -> 15.8.  Nothing at 96 KB of B tiles (1 x 1 512 -> 192 at 45 x 45 23.8 -> 23.7) or 2 - 5 tiles per CTA (64 -> 128 stride 2
  // at 56 x 56, batch 48, 64, 128: 13.2, 15.3, 22.9 -> 22.8).  Outside the rule, forced: 128 KB 27.5 -> 27.0, three A stages of a
  // row-batched multiply 18.5 -> 18.4; 32-byte rows were slower when the rule was made (5 x 5 32 -> 96 35.9 -> 37.6, 7 x 7
  // stride 2 RGB 33.4 -> 34.0) and as kernels stand 5 x 5 32 -> 96 is the same, 16 -> 64 70.4 -> 61.9, 1 x 1 32 -> 256 24.4 -> 21.5.
  if (ctas == 1 && !p.halo && p.splits == 1 && p.n_tiles_n == 1 && p.dstride <= 1 && g.kind != GK_FC_WGRAD && g.kind != GK_CONV_WGRAD &&
      (p.mrep > 1 || (p.kdepth >= 64 && tiles >= 3LL * units)) && (long long)p.kb_total * p.b_bytes <= 112 * 1024 && p.kb_total * p.b_bytes + 4 * p.a_bytes <= 200 * 1024) {
    p.b_resident = 1;
    p.b_tile_bytes = p.b_bytes;
    p.b_res_bytes = p.kb_total * p.b_bytes;
    p.b_bytes = 0;
    stage_bytes = p.a_bytes;
    p.stages = (200 * 1024 - p.b_res_bytes) / stage_bytes;
    if (p.stages > MAX_STAGES) p.stages = MAX_STAGES;
  }
  // rows with a pitch that is no multiple of 8: staging buffers of the fused epilogue's stores
  p.nstg_off = 0;
  if (p.splits == 1 && !p.halo && ((g.gn & 7) != 0 || (g.kind == GK_CONV_WGRAD && (p.Cn & 7) != 0))) {
    int st = (200 * 1024 - p.b_res_bytes - EPI_WARPS * 32 * 36) / stage_bytes;
    if (st > MAX_STAGES) st = MAX_STAGES;
    if (st < 2) return false;
    p.stages = st;
    p.nstg_off = p.b_res_bytes + st * stage_bytes;
  }
  if (p.halo) {
    p.splits = 1;
    p.kb_per_split = p.kb_total;
  }
  // producer warps: the largest count <= PROD_WARPS that divides the number of stages
  if (p.stages == 5 || p.stages == 7) p.stages -= 1;
  p.nissue = p.halo == 1 ? 2 : 1;
  p.nprod = 1;
  for (int d = 2; d <= PROD_WARPS - (p.nissue - 1); ++d)
    if (p.stages % d == 0) p.nprod = d;
  p.nbuf = 512 / p.bn;
  if (p.nbuf > MAX_TBUF) p.nbuf = MAX_TBUF;
  // epilogue groups: as many as leave no warp without a chunk and one spare accumulator buffer; without the spare
  // one where the epilogue of a plain multiply is the bound and no MMA waits for long (single CTAs, 8192 x 8192 at
  // K = 256 / 512 / 1024 40.5 -> 39.8, 46.3 -> 44.7, 63.3 -> 61.8 us, the gradient above 64.8 -> 59.6 us;
  // convolutions of the same depth are 1 - 4 % slower that way)
  const bool short_fc = ctas == 1 && g.kind <= GK_FC_WGRAD && g.gk <= PAIR_MIN_K;
  p.egroups = 1;
  for (int gq = 2; gq <= 4; gq *= 2)
    if (EPI_PER_Q / gq <= p.bn / 32 && p.nbuf >= gq + (short_fc ? 0 : 1)) p.egroups = gq;
  p.nbuf = p.nbuf / p.egroups * p.egroups;     // a buffer always returns to the same group
  p.one_commit = 0;
  if (p.halo == 1 && p.stages >= p.nbuf) {
    p.one_commit = 1;
    p.stages = p.nbuf;
    p.nprod = 1;
    for (int d = 2; d <= PROD_WARPS - (p.nissue - 1); ++d)
      if (p.stages % d == 0) p.nprod = d;
  }
  // convolution outputs are spatially structured (borders, images): contiguous item ranges make the
  // first tile of every CTA an even sample of the tensor for the speculative shift
  p.blocked = (g.kind == GK_CONV_FWD || g.kind == GK_CONV_DGRAD) ? 1 : 0;
  p.items = tiles * p.splits * (p.dstride > 1 ? p.nph_r * p.nph_s : 1);
  if (p.items >= (1LL << 30)) return false;      // the kernel counts items in 32 bits
  // the copies an instance issues have the rank and mode of its maps: anything else is a planning error
  if (p.halo == 1 && (sb.nd != (p.mode >= 1 ? 3 : 2) || sa.nd != 4 || sa.im2col)) return false;
  if (!p.halo && (g.kind == GK_CONV_FWD || g.kind == GK_CONV_DGRAD) &&
      (sb.nd != (p.mode >= 1 ? 3 : 2) || sa.nd != 4 || sa.im2col != p.i2c))
    return false;
  if (!p.halo && g.kind == GK_CONV_WGRAD && (sa.nd != (p.i2c ? 2 : 4) || sb.nd != 4 || sb.im2col != p.i2c)) return false;
  if (p.i2c && p.mode < 1) return false;
  if (!encode(ctx, &ma, sa) || !encode(ctx, &mb, sb)) return false;
  return true;
}

}  // namespace


int niti_tc_timeout_probe(niti_ctx *ctx, cudaStream_t st) {
  timeout_probe_kernel<<<1, 32, 0, st>>>(ctx->d_status);
  ctx->launches++;
  NITI_CUDA_TRY(ctx, cudaGetLastError());
  return NITI_OK;
}

// CTAs (CTAS = 1) or CTA pairs (CTAS = 2) that can be resident at the same time.  SMs pair up inside a
// GPC, so the number of pairs can be below sm_count / 2; a persistent grid larger than that would run
// a second, short wave.
// Dynamic shared-memory limit of the kernel: once per context, and always the most the device allows
// beside the kernel's static shared memory (see niti_ctx::smem_optin for why not "what this launch needs").
template <int CTAS, int MODE, bool ONE>
static int tc_set_smem_limit(niti_ctx *ctx) {
  cudaFuncAttributes fa;
  NITI_CUDA_TRY(ctx, cudaFuncGetAttributes(&fa, tc_gemm_kernel<CTAS, MODE, ONE>));
  const size_t limit = ctx->smem_optin > fa.sharedSizeBytes ? ctx->smem_optin - fa.sharedSizeBytes : 0;
  NITI_CUDA_TRY(ctx, cudaFuncSetAttribute(tc_gemm_kernel<CTAS, MODE, ONE>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)limit));
  ctx->tc_attr_smem[CTAS + 2 * MODE + 6 * ONE] = limit;
  return NITI_OK;
}

template <int CTAS>
static int tc_units(niti_ctx *ctx) {
  int &cached = ctx->tc_units[CTAS];
  if (cached) return cached;
  cached = ctx->sm_count / CTAS;
  if (CTAS == 2) {
    cudaLaunchConfig_t cfg;
    memset(&cfg, 0, sizeof(cfg));
    cfg.gridDim = dim3((unsigned)(ctx->sm_count / 2 * 2), 1, 1);
    cfg.blockDim = dim3(NUM_THREADS, 1, 1);
    cfg.dynamicSmemBytes = 200 * 1024;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = 2;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    (void)tc_set_smem_limit<2, 0, false>(ctx);
    int n = 0;
    if (cudaOccupancyMaxActiveClusters(&n, tc_gemm_kernel<2, 0, false>, &cfg) == cudaSuccess && n > 0 && n < cached) cached = n;
    else (void)cudaGetLastError();
  }
  return cached;
}

template <int CTAS, int MODE, bool ONE>
static int launch_tc_as(niti_ctx *ctx, cudaStream_t st, const TcParams &p, const CUtensorMap &ma, const CUtensorMap &mb, const CUtensorMap &mc,
                     int32_t *acc, WsHeader *hdr, const RoundSpec &r) {
  size_t smem = (size_t)p.stages * (p.a_bytes + p.b_bytes) + (size_t)p.b_res_bytes + 1024;
  if (p.red) smem = (size_t)p.red_off + RED_BYTES + 1024;
  if (p.nstg_off > 0) smem = (size_t)p.nstg_off + (size_t)EPI_WARPS * 32 * 36 + 1024;
  size_t &attr_smem = ctx->tc_attr_smem[CTAS + 2 * MODE + 6 * ONE];
  if (!attr_smem) {
    const int rcs = tc_set_smem_limit<CTAS, MODE, ONE>(ctx);
    if (rcs != NITI_OK) return rcs;
  }
  if (smem > attr_smem) return niti_fail(ctx, NITI_ERR_SHAPE, "tensor-core kernel: stage buffers exceed the shared memory of an SM");
  cudaLaunchConfig_t cfg;
  memset(&cfg, 0, sizeof(cfg));
  cfg.gridDim = dim3((unsigned)(ctx->sm_count / CTAS * CTAS), 1, 1);
  cfg.blockDim = dim3(NUM_THREADS, 1, 1);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = CTAS;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;     // (see niti_enter)
  attr[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.numAttrs = 2;
  const int units = tc_units<CTAS>(ctx);
  long long grid = (p.items < units ? p.items : units) * CTAS;
  cfg.gridDim = dim3((unsigned)grid, 1, 1);
  TcParams q = p;
  {
    const int gunits = (int)(grid / CTAS);
    q.blk_per = (int)(p.items / gunits);
    q.blk_extra = (int)(p.items % gunits);
    // (a CTA with a single tile has all its epilogue warps on that tile)
    if (p.items <= gunits) q.egroups = 1;
    const int eg = p.halo == 2 ? 1 : q.egroups;
    q.k_wpq = EPI_PER_Q / eg;
    const int chunks_all = p.bn / 32;
    q.k_wpq_active = p.halo == 2 ? EPI_PER_Q : (chunks_all < q.k_wpq ? chunks_all : q.k_wpq);
    q.k_epi_active = 4 * q.k_wpq_active;
    int cols = 32;
    while (cols < p.nbuf * p.bn) cols <<= 1;
    q.k_tmem_cols = cols;
    // (dividends are items, tiles, grid positions or k-blocks, all below 2^31: plan() refuses others)
    q.d_w = make_div(p.w_tiles);
    q.d_h = make_div(p.h_tiles);
    q.d_n = make_div(p.n_tiles_n);
    q.d_split = make_div(p.splits);
    if (p.raster_g > 0) {
      q.last_group = (p.m_units - 1) / p.raster_g;
      q.d_group = make_div((long long)p.raster_g * p.n_tiles_n);
      q.d_units = make_div(p.raster_g);
      q.d_last = make_div(p.m_units - q.last_group * p.raster_g);
    }
    q.d_chunks = make_div(p.n_chunks);
    q.d_S = make_div(p.S);
    q.d_cc = make_div(p.c_chunks);
    q.d_phases = make_div((long long)p.nph_r * p.nph_s);
    q.d_phase_s = make_div(p.nph_s);
    for (int v = p.Wt; v > 1; v >>= 1) q.wt_shift++;
    for (int v = p.Ht; v > 1; v >>= 1) q.ht_shift++;
    for (int v = q.k_wpq; v > 1; v >>= 1) q.k_wpq_shift++;
    // how the rows of the output lie and what is done to them
    q.row_kind = p.dstride > 1 ? ROWS_PHASES : p.halo ? ROWS_HALO
                 : p.kind == GK_CONV_WGRAD ? ROWS_WGRAD
                 : (p.kind == GK_CONV_FWD || p.kind == GK_CONV_DGRAD) && !p.i2c ? ROWS_BOXES : ROWS_PLAIN;
    const unsigned bits = (unsigned)p.gn | (unsigned)(uintptr_t)r.out | (r.mask ? (unsigned)(uintptr_t)r.mask : 0u) | 32u |
                          (p.kind == GK_CONV_WGRAD ? (unsigned)p.Cn : 0u);
    q.io_unit = (int)(bits & (0u - bits));
    if (q.io_unit < 32) {
      const unsigned out_bits = (unsigned)p.gn | (unsigned)(uintptr_t)r.out | 16u | (p.kind == GK_CONV_WGRAD ? (unsigned)p.Cn : 0u);
      q.io_unit = (int)(out_bits & (0u - out_bits));          // (gate bytes are read at any alignment)
    }
    const bool narrow = q.io_unit < 32;
    q.form = p.mrep > 1 ? (narrow ? (r.relu ? LEAN_BATCHED_NARROW_RELU : LEAN_BATCHED_NARROW) : r.relu ? LEAN_BATCHED_RELU : LEAN_BATCHED)
             : narrow ? (r.relu ? LEAN_NARROW_RELU : r.mask ? LEAN_NARROW_MASK : LEAN_NARROW)
             : p.update ? LEAN_UPDATE : p.pool ? LEAN_POOL : r.relu ? LEAN_RELU : r.mask ? LEAN_MASK : LEAN_PLAIN;
  }
  // per call site (keyed by the address of its bit-width scalar): the error of the last speculative estimate
  int32_t *slot = nullptr;
  if (r.b_out && ctx->d_spec_tab) {
    const uintptr_t key = (uintptr_t)r.b_out >> 2;
    slot = ctx->d_spec_tab + 2 * (size_t)((key ^ (key >> 13)) % NITI_SPEC_SLOTS);
    q.spec_tag = (int)(unsigned)(key | 1u);
  }
  NITI_CUDA_TRY(ctx, cudaLaunchKernelEx(&cfg, tc_gemm_kernel<CTAS, MODE, ONE>, ma, mb, mc, q, acc, hdr, ctx->d_status, r.out, r.mask,
                                        r.s_a, r.s_w, r.s_out, r.b_out, slot, r.pool_out));
  ctx->launches++;
  ctx->tc_launches++;
  if (CTAS == 2) ctx->tc2_launches++;
  if (p.b_resident) ctx->res_launches++;
  return NITI_OK;
}

static int launch_tc(niti_ctx *ctx, cudaStream_t st, const TcParams &p, const CUtensorMap &ma, const CUtensorMap &mb, const CUtensorMap &mc,
                     int32_t *acc, WsHeader *hdr, const RoundSpec &r) {
  auto go = [&](auto mode, auto one) {
    constexpr int MODE = decltype(mode)::value;
    constexpr bool ONE = decltype(one)::value;
    return p.ctas == 2 ? launch_tc_as<2, MODE, ONE>(ctx, st, p, ma, mb, mc, acc, hdr, r)
                       : launch_tc_as<1, MODE, ONE>(ctx, st, p, ma, mb, mc, acc, hdr, r);
  };
  auto pick = [&](auto mode) {
    return p.single_wave && p.epi_mode == EPI_SPECULATE ? go(mode, std::true_type{}) : go(mode, std::false_type{});
  };
  if (p.mode == 2) return pick(std::integral_constant<int, 2>{});
  if (p.mode == 1) return pick(std::integral_constant<int, 1>{});
  return pick(std::integral_constant<int, 0>{});
}

// Profiling event of a launch.  On a stream that is being captured the record becomes an event-record
// node of the graph (cudaEventRecordExternal), so that every replay of the graph times its launches
// where they run; a plain record there would only add a dependency.
static void prof_record(cudaEvent_t ev, cudaStream_t st) {
  cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
  if (cudaStreamIsCapturing(st, &cap) == cudaSuccess && cap == cudaStreamCaptureStatusActive)
    cudaEventRecordWithFlags(ev, st, cudaEventRecordExternal);
  else
    cudaEventRecord(ev, st);
}

// Cycles of one k-block of a tile: the MMAs (bound by their math or by the shared-memory reads of their operands) or
// the operand copies (measured: about 84 bytes per clock into one SM, 9000 into all of them; never below 400 cycles for
// 128 contraction elements however narrow the tile).
static double kblock_cycles(const TcParams &p, int ctas, int bn, long long ctas_running) {
  const double mma = bn / 2.0, smem = 32.0 + bn / (4.0 * ctas), bytes = (128.0 + (double)bn / ctas) * p.kdepth;
  double c = p.ksteps * (mma > smem ? mma : smem);
  if (c < bytes / 84.0) c = bytes / 84.0;
  if (c < bytes * ctas_running / 9000.0) c = bytes * ctas_running / 9000.0;
  return c < 100.0 * p.ksteps ? 100.0 * p.ksteps : c;
}
// A multiply of at most one tile per SM: an unsplit plan whose every CTA (pair) has one tile rounds in its own epilogue
// with an exact shift, in one launch.  Splitting the contraction shortens the main loop but costs a zeroed scratch, the
// reduce copies and a finishing launch over the int32 sums; pairs of CTAs cost 0.8 us more set-up than single ones.  (The
// constants of the model were measured on earlier kernels: a split's 3.5 us + 5 us per million outputs when two kernels
// finished it, several waves' when their agreement took twice as long.)  What it decides, as kernels stand (graph replay, without
// one-wave plans -> with them, forward / error / gradient, where the plan changes): 256 images of 4 x 4, 512 -> 512 channels, 27.9
// -> 18.8 / 24.9 -> 17.6 / 25.5 -> 16.7 us; 100 of 9 x 9, 96 -> 160, 17.7 -> 10.0 / 17.9 -> 12.2; 64 of 7 x 7, 256 -> 512, 26.1 ->
// 12.4 / 19.3 -> 17.0 / 20.8 -> 14.5; 128 of 8 x 8, 128 -> 256, 20.1 -> 11.0 / 19.8 -> 13.6; 256 of 2 x 2, 512 -> 512, 16.5 ->
// 16.2 / 17.1 -> 17.7 / 21.2 -> 11.7; 32 of 14 x 14, 256 -> 256, 20.6 -> 12.3 / 21.5 -> 13.7; 77 of 11 x 11, 64 -> 192, 19.0 ->
// 9.1 / 16.5 -> 12.0; 30 of 13 x 13, 192 -> 384, 28.0 -> 11.8 / 21.0 -> 14.7; 5 x 5, 64 of 8 x 8, 256 -> 256, 21.1 -> 20.7 / 21.8 ->
// 21.9 / 22.9 -> 16.2; fully connected, forward / backward, 1024^3 15.6 -> 10.6 / 31.6 -> 20.3, 4096 x 1000 x 512 11.2 / 42.4 ->
// 29.9, 2048 x 2048 x 512 9.7 / 37.5 -> 25.0, 512 x 4096 x 1024 20.5 -> 11.3 / 28.8 -> 25.1, 1500 x 700 x 3000 25.4 -> 20.8 / 45.3 ->
// 36.9, 256 x 4096 x 4096 19.5 -> 17.1 / 42.5 -> 38.0: of 53 multiplies one is 3.5 % slower, none of the others by more than
// two measurements differ.  (Splits that form a cluster and add their partial tiles through distributed shared memory were
// built and measured: 24.3 - 25.0 us against 20.7 us unsplit on the first of these; the agreement over twice as many CTAs and
// the exchange cost what the shorter main loop saves.)
static bool pick_one_wave(niti_ctx *ctx, const GemmProblem &g, const TcParams &p, int &ctas, int &bn) {
  const int units = p.ctas == 2 ? tc_units<2>(ctx) : tc_units<1>(ctx);
  if (p.halo || p.mrep > 1 || p.dstride > 1 || p.items > 4LL * units) return false;
  const long long waves = (p.items + units - 1) / units, running = (p.items < units ? p.items : units) * p.ctas;
  double best = (double)waves * (p.kb_per_split * kblock_cycles(p, p.ctas, p.bn, running) + (waves > 1 ? 3000.0 : 0.0)) +
                (p.ctas == 2 ? 1500.0 : 0.0) +
                (p.splits > 1 ? 6500.0 + 0.0095 * (double)g.gm * (double)g.gn : (waves > 1 ? 3500.0 : 0.0));
  best *= 0.97;
  const int cols = g.kind == GK_CONV_WGRAD ? p.Cn : (int)g.gn, taps = g.kind == GK_CONV_WGRAD ? g.R * g.S : 1;
  const bool boxes = (g.kind == GK_CONV_FWD || g.kind == GK_CONV_DGRAD) && !p.i2c;
  const long long m128 = boxes ? (long long)p.w_tiles * p.h_tiles * p.b_tiles : (g.gm + BM - 1) / BM;
  bool found = false;
  for (int c = 1; c <= 2; ++c) {
    if (c == 2 && g.gm < 2 * BM) break;
    const long long mu = (m128 + c - 1) / c, cap = c == 2 ? tc_units<2>(ctx) : tc_units<1>(ctx);
    for (int nt = (cols + 255) / 256; nt <= (cols + 31) / 32 && mu * nt * taps <= cap; ++nt) {
      const int w = round_up32((cols + nt - 1) / nt);
      if ((cols + w - 1) / w != nt) continue;
      const double t = p.kb_total * kblock_cycles(p, c, w, mu * nt * taps * c) + (c == 2 ? 1500.0 : 0.0);
      if (t < best) { best = t * 0.99; ctas = c; bn = w; found = true; }
    }
  }
  return found;
}

// Launches finish_split_kernel where the sums fit the registers of one block per SM; NITI_ERR_SHAPE otherwise.
static int launch_finish(niti_ctx *ctx, cudaStream_t st, const int32_t *acc, long long n, WsHeader *hdr, int splits,
                         const RoundSpec &r) {
  const long long nvec = n >> 2;
  const int most = ctx->sm_count < NITI_AGREE_MAX ? ctx->sm_count : NITI_AGREE_MAX;
  if ((n & 3) || splits > NITI_MAX_SPLITS - NITI_AGREE_WORDS || nvec > (long long)most * FIN_THREADS * 8 ||
      (((uintptr_t)r.out | (uintptr_t)r.update_w | (uintptr_t)r.mask) & 3))
    return NITI_ERR_SHAPE;
  long long blocks = (nvec + FIN_THREADS - 1) / FIN_THREADS;
  if (blocks > most) blocks = most;
  const long long per = (nvec + blocks * FIN_THREADS - 1) / (blocks * FIN_THREADS);
  auto go = [&](auto kernel) {
    return niti_launch(st, (unsigned)blocks, FIN_THREADS, 0, kernel, acc, (int)nvec, hdr, splits, ctx->d_status, r.out, r.update_w, r.mask, r.relu, r.mbits,
                              r.round_mode, r.s_a, r.s_w, r.s_out, r.b_out, ctx->patience);
  };
  NITI_CUDA_TRY(ctx, per <= 1 ? go(finish_split_kernel<1>) : per <= 2 ? go(finish_split_kernel<2>)
                     : per <= 4 ? go(finish_split_kernel<4>) : go(finish_split_kernel<8>));
  ctx->launches++;
  return NITI_OK;
}

// Is no operand (nor the gate) in the storage of an output?  Then outputs may be stored before all operands have been read,
// and stored again: a CTA's first tile during the agreement, all of them where a guess was wrong.
static bool may_store_twice(const GemmProblem &g, const RoundSpec &r) {
  const long long x = (long long)g.B * g.H * g.W * g.Ci, y = (long long)g.B * g.Ho * g.Wo * g.Co;
  const long long out_bytes = g.gm * g.gn;
  long long n0, n1;
  switch (g.kind) {
    case GK_FC_FWD: n0 = (long long)g.M * g.K; n1 = (long long)g.N * g.K; break;
    case GK_FC_DGRAD: n0 = (long long)g.M * g.N; n1 = (long long)g.N * g.K; break;
    case GK_FC_WGRAD: n0 = (long long)g.M * g.N; n1 = (long long)g.M * g.K; break;
    case GK_CONV_FWD: n0 = x; n1 = (long long)g.Co * g.R * g.S * g.Ci; break;
    case GK_CONV_DGRAD: n0 = y; n1 = (long long)g.Co * g.R * g.S * g.Ci; break;
    default: n0 = y; n1 = x; break;
  }
  auto apart = [](const void *a, long long na, const void *b, long long nb) {
    const uintptr_t u = (uintptr_t)a, v = (uintptr_t)b;
    return !a || !b || u + (uintptr_t)na <= v || v + (uintptr_t)nb <= u;
  };
  auto output_apart = [&](const int8_t *out, long long n) {
    // (a padded or widened copy is read in place of the operand, whose extents are then others)
    return (g.q0 || apart(out, n, g.p0, n0)) && (g.q1 || apart(out, n, g.p1, n1)) && apart(out, n, r.mask, out_bytes);
  };
  return output_apart(r.out, out_bytes) && output_apart(r.pool_out, out_bytes / 4);
}

int niti_tc_gemm(niti_ctx *ctx, cudaStream_t st, const GemmProblem &g_in, const RoundSpec &r_in, int32_t *acc,
                 WsHeader *hdr, bool *fused, bool *pooled, bool shard_ok, bool *updated) {
  GemmProblem g = g_in;
  g.in_place = !may_store_twice(g_in, r_in);
  TcParams p;
  CUtensorMap ma, mb, mc;
  memset(&mc, 0, sizeof(mc));
  RoundSpec r = r_in;
  *fused = false;
  if (pooled) *pooled = false;
  if (updated) *updated = false;
  // engine 0: pairs of CTAs (cta_group::2) when there are enough 256-row tiles to fill the GPU.
  // Test switches: 2 / 3 force the single-CTA / paired kernel, 4 keeps the int32 spill epilogue.
  // Test switches: 5 disables the halo mode of small-channel convolutions.
  // (columns of one tap of a convolution's weight gradient start at multiples of the channel count)
  const bool aligned = (g.gn & 31) == 0 && ((uintptr_t)r.out & 31) == 0 && ((uintptr_t)r.mask & 31) == 0 &&
                       (g.kind != GK_CONV_WGRAD || (g.Ci & 31) == 0);
  bool planned = false;
  if ((g.kind == GK_CONV_FWD || g.kind == GK_CONV_DGRAD || g.kind == GK_CONV_WGRAD) && ctx->engine != 3 &&
      ctx->engine != 5)
    planned = plan(ctx, g, 1, PLAN_HALO, aligned, 0, acc, p, ma, mb, mc);
  if (!planned && g.kind == GK_FC_FWD && ctx->engine != 3)      // row-batched mode of short contractions
    planned = plan(ctx, g, 1, PLAN_BATCHED, aligned, 0, acc, p, ma, mb, mc);
  // Pairs halve the operand traffic per MMA, and couple two SMs' epilogues to one accumulator.  With a short
  // contraction the epilogue is the bound (about 3 - 4 k cycles per tile against 560 per k-block of 128), and two
  // CTAs that drain their own tiles are ahead: gradient of 4096 x 25088 weights at batch 64 92 -> 65 us, 8192 x 8192
  // at K = 256 / 512 / 1024 / 2048 54 -> 41, 55 -> 46, 64 -> 63, 90 -> 102 us; convolutions with K = 128 69.5 -> 52.4,
  // 1152 25.6 -> 23.7, 2304 82 -> 92 us; strided errors (K of one phase) with K = 576 40.1 -> 36.2 us.
  const long long k_tile = g.gk / (g.kind == GK_CONV_DGRAD ? (long long)g.stride * g.stride : 1);
  if (!planned && ctx->engine != 2 && g.gm >= 2 * BM && (ctx->engine == 3 || k_tile > PAIR_MIN_K)) {
    planned = plan(ctx, g, 2, PLAN_ANY, aligned, 0, acc, p, ma, mb, mc);
    // (pairs halve the operand traffic per MMA; they are kept unless they would leave more than a
    // third of the GPU idle)
    if (planned && ctx->engine != 3 && p.items * 3 < (long long)(ctx->sm_count / 2) * 2) planned = false;
  }
  if (!planned) {
    if (ctx->engine == 3) return NITI_ERR_SHAPE;
    if (!plan(ctx, g, 1, PLAN_ANY, aligned, 0, acc, p, ma, mb, mc)) return NITI_ERR_SHAPE;
  }
  if (ctx->engine == 0 && !ctx->reduce_fn && r.out) {
    int c = 0, w = 0;
    if (pick_one_wave(ctx, g, p, c, w)) {
      TcParams p1;
      CUtensorMap a1, b1, c1;
      if (plan(ctx, g, c, PLAN_ANY, aligned, w, acc, p1, a1, b1, c1)) {
        p = p1;
        ma = a1;
        mb = b1;
      }
    }
  }
  {
    // expected ratio between the max of the whole tensor (N values) and the max of the first tile of
    // every CTA (n values) for roughly Gaussian sums: sqrt(ln N / ln n)
    const int units = p.ctas == 2 ? tc_units<2>(ctx) : tc_units<1>(ctx);
    const double n_all = (double)g.gm * (double)g.gn;
    const double frac = p.items > units ? (double)units / (double)p.items : 1.0;
    const double n_s = n_all * frac;
    double f = (n_s > 16.0 && frac < 1.0) ? sqrt(log(n_all) / log(n_s)) : 1.0;
    p.spec_mul256 = (unsigned)(f * 256.0 + 0.5);
    const double n_own = n_all / ((double)p.items * p.ctas);
    const double f_own = n_own > 16.0 ? sqrt(log(n_all) / log(n_own)) : 1.0;
    p.trial_mul256 = !g.in_place ? (unsigned)(f_own * 256.0 + 0.5) : 0u;
  }
  // data parallelism (niti_set_reduce_hook): the max magnitude is combined over the ranks between the
  // two launches, so there is always a second launch; weight gradients keep their int32 sums
  const bool dp = ctx->reduce_fn != nullptr, dp_sum = dp && niti_is_wgrad(g.kind);
  p.single_wave = (!dp && p.items * p.ctas <= NITI_AGREE_MAX && p.items <= (p.ctas == 2 ? tc_units<2>(ctx) : tc_units<1>(ctx)) && p.spec_mul256 == 256) ? 1 : 0;
  p.patience = ctx->patience;
  p.mbits = r.mbits;
  p.round_mode = r.round_mode;
  p.relu = r.relu;
  // (an output in the storage of an operand or of the gate: rounded after the whole multiply, where not in one wave, whose
  // CTAs store when all have read.  A strided error with phases that no window reaches clears its output beforehand.)
  const bool sums_first = g.in_place && (!p.single_wave || p.dstride > 1);
  p.epi_mode = (p.splits > 1 || p.halo == 2) ? EPI_ATOMIC : ((ctx->engine == 4 || dp_sum || !r.out || sums_first) ? EPI_SPILL : EPI_SPECULATE);
  if (p.dstride > 1 && (p.nph_r < p.dstride || p.nph_s < p.dstride)) {
    // filter smaller than the stride: no window reaches the input pixels of the other phases
    if (p.epi_mode == EPI_SPILL) NITI_CUDA_TRY(ctx, cudaMemsetAsync(acc, 0, sizeof(int32_t) * (size_t)(g.gm * g.gn), st));
    else NITI_CUDA_TRY(ctx, cudaMemsetAsync(r.out, 0, (size_t)(g.gm * g.gn), st));
    ctx->launches++;
  }
  const bool sums = p.epi_mode == EPI_ATOMIC;
  int rc = niti_clear(ctx, st, sums ? acc : nullptr, sums ? sizeof(int32_t) * (size_t)(g.gm * g.gn) : 0, &p.next);
  if (rc != NITI_OK) return rc;
  // Fused 2 x 2 max-pool: the fused epilogue of a forward convolution with ReLU also stores the pooled
  // tile when every pooling window lies inside one warp's 32 pixels (8 x 16 pixel tiles of the
  // resident-weights mode, or pixel boxes at most 16 wide and at least 2 high) and the rows are whole,
  // 32-byte aligned chunks.  Otherwise the caller runs the pooling kernel.
  p.pool = 0;
  if (pooled && r.pool_out && g.kind == GK_CONV_FWD && r.relu && !r.mask && p.epi_mode == EPI_SPECULATE &&
      p.mrep == 1 && (p.PW % 2) == 0 && (p.PH % 2) == 0 && (g.gn % 32) == 0 && ((uintptr_t)r.out & 31) == 0 &&
      ((uintptr_t)r.pool_out & 31) == 0 && r.mbits == 7) {
    if (p.halo == 1) { p.pool = 1; p.pool_xh = 8; }
    else if (!p.halo && p.Wt >= 2 && p.Wt <= 16 && p.Ht >= 2) { p.pool = 1; p.pool_xh = p.Wt; }
    *pooled = p.pool != 0;
  }
  // Weight update inside the epilogue (Section 3.3): a weight gradient whose epilogue
  // rounds by itself subtracts the rounded values from the weights in place of storing them.  A
  // speculative pass must not touch the weights (a wrong guess could not be taken back), so the update
  // is fused only where the shift is exact when the stores happen: single-wave launches.  (Measured
  // and not kept for the other launches: a first pass for the bit-width alone followed by a rounding
  // pass that updates, 198 us against 185 us for the 4096 x 25088 layer at batch 64, when its gradient ran on CTA
  // pairs; the three launches now take 138 us with the error.)
  p.update = 0;
  if (updated && r.update_w && (g.kind == GK_FC_WGRAD || (g.kind == GK_CONV_WGRAD && (g.Ci & 31) == 0)) &&
      p.epi_mode == EPI_SPECULATE && p.single_wave && p.mrep == 1 && !p.halo && !r.mask && !r.relu && (g.gn % 32) == 0 &&
      ((uintptr_t)r.update_w & 31) == 0) {
    p.update = 1;
    p.trial_mul256 = 0;
    r.out = r.update_w;
    *updated = true;
  }
  const bool prof = ctx->profile_on && ctx->prof_ev && ctx->prof_used < NITI_PROF_MAX;
  if (prof) prof_record(ctx->prof_ev[2 * ctx->prof_used], st);
  rc = launch_tc(ctx, st, p, ma, mb, mc, acc, hdr, r);
  if (rc != NITI_OK) return rc;
  niti_header_passed_on(ctx, p.next);
  p.next = nullptr;
  if (p.epi_mode == EPI_SPECULATE && p.single_wave) {
    *fused = true;                     // exact shift, scalars published by this launch: no second one
  } else if (p.epi_mode == EPI_SPECULATE) {
    // publishes b and the exponent; recomputes with the true bit-width only if the guess was low
    if (dp) {
      rc = niti_reduce(ctx, st, &hdr->maxabs32, 1, NITI_REDUCE_MAX_U32);
      if (rc != NITI_OK) return rc;
    }
    p.epi_mode = EPI_KNOWN_B;
    rc = launch_tc(ctx, st, p, ma, mb, mc, acc, hdr, r);
    if (rc != NITI_OK) return rc;
    *fused = true;
  }
  if (prof) {
    prof_record(ctx->prof_ev[2 * ctx->prof_used + 1], st);
    ctx->prof_ops[ctx->prof_used] = 2.0 * (double)g.gm * (double)g.gn * (double)g.gk;
    ctx->prof_used++;
  }
  if (p.epi_mode == EPI_ATOMIC) {
    // (weight gradients under data parallelism: the sums over the ranks first, then their max)
    if (dp_sum) return niti_reduce_after_gemm(ctx, st, g.kind, acc, g.gm * g.gn, hdr, shard_ok);
    if (!dp && r.out && (rc = launch_finish(ctx, st, acc, g.gm * g.gn, hdr, p.splits, r)) != NITI_ERR_SHAPE) {
      *fused = true;
      if (updated) *updated = r.update_w != nullptr;
      return rc;
    }
    rc = niti_launch_maxabs(ctx, st, acc, g.gm * g.gn, hdr, p.splits);
    if (rc != NITI_OK || !dp) return rc;
    return niti_reduce(ctx, st, &hdr->maxabs32, 1, NITI_REDUCE_MAX_U32);
  }
  if (p.epi_mode == EPI_SPILL && dp) return niti_reduce_after_gemm(ctx, st, g.kind, acc, g.gm * g.gn, hdr, shard_ok);
  return NITI_OK;
}
