// Dense regrouping on the tensor cores: the layer as an implicit GEMM over zero-inserted weights,
// D[pixel, filter] = sum over (tap, channel) of A_tap[pixel, channel] * W_tap[channel, filter], on
// tcgen05.mma with the accumulators in Tensor Memory.
//
// Why it exists beside the pattern-sparse kernel: it does 9 / (4 x keep) times the multiply-adds (for
// fp32 storage six times that), but the tensor pipe delivers ~2000 TFLOP/s where the FP32 pipe has 74,
// of which the sparse kernel's per-kernel jump leaves 15-20.
//
// Precision.  fp16 storage: products are exact in fp32, sums are fp32.  fp32 storage: every activation
// and weight is cut into three bf16 pieces, x = x1 + x2 + x3 exactly (from 2^-110 up; 8 + 8 + 8 bits, rounded to nearest
// so that the pieces' signs are random), and six of the nine piece products are formed:
//   main  x1 w1;   cross  x1 w2, x2 w1, x2 w2, x1 w3, x3 w1
// The three left out are below 2^-24 of the product together.  The tensor core adds with truncation
// (measured: one round-toward-zero per instruction at the accumulator's exponent; 288 additions of
// 16 products leave 1e-5), so the main sums never stay there for more than one channel step: after
// nine instructions the epilogue warps add them to fp32 registers (rounded to nearest) while the cross
// products of the next step run.  The cross sums are 2^-8 as large and stay in Tensor Memory.
//
// Mapping.
//  * Positions.  An output map is a run of rows of `pitch` positions (its columns, then at least one
//    zero column, which is the padding right of one row and left of the next) closed by one zero row
//    (the padding below one image and above the next); maps wider than a strip are cut into column
//    strips that carry both neighbours.  The batch is one long line of positions, an MMA tile is 128
//    consecutive ones, and a tap is the same line shifted by a constant.
//  * A operand.  Shared memory holds, per 8 channels, one 16-byte row per position (K-major, no
//    swizzle, 8-row core matrices back to back), so position p is at p x 16 bytes and ANY shift is a
//    descriptor start address: one staged copy serves all nine taps.  Stride 2 stages the four
//    row / column parity planes and a fused 2x2 max-pool the two row parity planes, each a line of the
//    same pitch; the taps then pick plane and shift.
//  * B operand.  Weights in the same row format (filter = row), per (16-channel step, tap, 8 channels,
//    piece) all filters' rows back to back: any range of filters is one bulk copy.  Taps outside the
//    union of the layer's patterns are neither stored nor multiplied.
//  * Cost of one MMA of 128 x N x 16: max(N / 2, 32 + N / 4) cycles (measured; the second term is its
//    operands at 128 bytes a cycle from shared memory).  Pieces of the weights are therefore stacked
//    along N where one A operand meets several of them.
//  * Warps: 8 epilogue warps, one that issues the MMAs, one that streams weights through a ring, and
//    either 10 that load activations from NCHW, convert and store them, or one that copies them where they
//    come as position rows (below).  One persistent CTA per SM.
//  * Position rows.  Between the layers of a stack, and where the caller has memory for them, activations
//    lie in global memory as the tensor core reads them, split into pieces already: bulk copies replace
//    the producers' loads and conversions (256->256 56x56 fp32 N=1: 37 us against 33).
//  * Few tiles: channel steps are cut into parts that different CTAs take.  Up to eight CTAs of a tile form
//    a cluster and add their sums up through distributed shared memory, in rank order; otherwise partial
//    sums meet in the caller's workspace (16-byte vector reductions, a ticket per warp's part; the last
//    one finishes).
//  * Instruction caches.  The roles run different code side by side, so every loop is kept short: the
//    epilogue unrolled over its registers took 10 us a tile to fetch, a wait loop unrolled by the compiler
//    half of the kernel's speed.
//  * What bounds it: the tensor pipe in large fp32 launches (512->512 14x14 N=64: 589 us in the sparse
//    kernel, 312 here); with 64 filters or few channels the epilogue; at one image a fixed 9-10 us of
//    launch, first copies and exchange, then the weight stream (36 bytes a cycle and SM from L2).
//  * Every wait is bounded; one that runs out records its id in the status word, the role stops
//    working, and all roles meet at the common exit where Tensor Memory is released.
#include <cuda_fp16.h>

#include <algorithm>
#include <atomic>
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <mutex>
#include <type_traits>

#include "pconv_internal.h"

namespace pconv {
namespace {

typedef unsigned long long u64;

constexpr int kMaxA = 4;                  // activation stages (one 16-channel step each)
constexpr int kMaxB = 24;                 // weight slots
constexpr int kMaxT = 4;                  // 128-position tiles of a work item
constexpr int kHeader = 1024;             // barriers, Tensor Memory address, bias of a filter tile
constexpr int kBiasOff = 512;
static_assert(16 * (kMaxA + kMaxB) + 32 + 4 + 16 <= kBiasOff, "barriers, Tensor Memory address, segments to redo");
constexpr uint32_t kSpinLimit = 1u << 20;
// Wait ids in the status word (the tiled kernel's are below 20): a free stage or slot, a filled one, accumulators.
constexpr int kWaitFree = 21, kWaitFull = 22, kWaitSums = 23;
constexpr uint32_t kWaitHintNs = 200;
constexpr int kSmemLimit = 227 * 1024;
constexpr int kTables = 5;                // load tables of the NCHW producers: segments s - 1 .. s + 3

// P8: the activations come in position rows (see stage_kernel) that bulk copies move; otherwise the
// producer warps convert them from NCHW.
template <bool HALF, bool P8>
struct Cfg {
  static constexpr int kEpiWarps = 8;
  static constexpr int kProdWarps = P8 ? 1 : 10;
  static constexpr int kMmaWarp = kEpiWarps;
  static constexpr int kBWarp = kEpiWarps + 1;
  static constexpr int kProdWarp0 = kEpiWarps + 2;
  static constexpr int kProdThreads = 32 * kProdWarps;
  static constexpr int kThreads = 32 * (kEpiWarps + 2 + kProdWarps);
  static constexpr int kPieces = HALF ? 1 : 3;
  static constexpr int kGroups = kEpiWarps / 4;     // warps that share a lane quadrant: column groups
};

struct DGeo {
  int n, h, w, c_in, c_out, h_out, w_out;   // h_out, w_out: of the stored map (pooled if `pool`)
  int pitch, cell_rows, cell_pos;    // positions of a row; rows and positions of a (image, strip) cell
  int strips, strip_w, ox;           // column strips, their width, column offset of position 0
  int n_cells;
  int sy, sx;                        // input rows / columns per position row / column
  int planes, plane_pos, lead;       // staged planes, positions of each, positions before an item's first
  int q_tot;                         // planes * plane_pos
  int vec, n_vec, vec_rows, vec_cols, row_planes;   // loads: pixels of one, loads of a channel, their grid
  int tiles, pool, mpos;             // MMA tiles of an item, fused pool, positions of an item
  int nt, n_ft, form3;               // filters of a tile (multiple of 16), filter tiles; fp32: see kernel
  int out_col, out_stride;           // fp32: columns the finished sums go to (0: over the main sums), tiles' distance
  int tile_cols, n_buf;              // Tensor Memory columns of a tile; accumulator sets (fp16)
  int rows;                          // filter rows in the weight stream (c_out rounded up to 16)
  int n_taps, tps, slots;            // taps stored; taps of a ring slot; slots of a channel step
  int k_steps, split;                // channel steps of a tile; whether a tile may be shared by CTAs
  int a_stages, b_slots, a_off, b_off, a_bytes, b_bytes;
  int relu;
  int n_tiles, grid;                 // (positions, filters) tiles, CTAs
  int cluster;                       // the CTAs of a tile are a thread-block cluster and exchange their sums directly
  int share, share_more, parts;      // a CTA's tiles or steps (the first share_more: one more); equal parts of a tile
  uint32_t cell_mul, pitch_mul;      // p / cell_pos and p / pitch by multiplication, then shifts (see fast_div)
  int cell_shift, pitch_shift;
  int in_plane_len, in_lead;         // P8 source: positions of a plane, positions before the batch's first
  int out_p8, out_pitch, out_cell_rows, out_sy, out_sx, out_plane_len, out_lead;   // P8 result: the next layer's rows
  int tap_off[kMaxT][9];             // start position of (tile, stored tap) inside a staged slab
};

__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
// One arrival for the whole warp once every lane has come here (an arrival of each thread costs a few
// cycles apiece: 320 of them took longer than staging the step itself).
__device__ __forceinline__ void warp_arrive(uint32_t bar, int lane) {
  __syncwarp();
  if (lane == 0) mbar_arrive(bar);
}
__device__ __forceinline__ void mbar_arrive_expect_tx(uint32_t bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint32_t bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(bar), "r"(parity), "r"(kWaitHintNs)
      : "memory");
  return ok != 0;
}
#ifdef PCONV_DEV
// Development build: the channel step whose activations one producer thread never reports, and the
// bound of every wait (see pconv_dev.h).
__device__ int g_withhold_step = -1;
__device__ unsigned g_spin_limit = kSpinLimit;
#define D_SPIN_LIMIT (*(volatile unsigned*)&g_spin_limit)
#define D_WITHHOLD_STEP (*(volatile int*)&g_withhold_step)
// CTA 0 leaves in the layer's trace words the cycles its roles waited and worked: MMA warp 0 all, 1 waiting
// for accumulators, 2 for activations, 3 for weights; producer thread 0: 4 all, 5 waiting for a free stage;
// weight stream 6 waiting for a free slot; epilogue thread 0: 7 waiting for accumulators, 8 taking main
// sums, 9 finishing.
#define T_DECL long long tw_[10] = {0, 0, 0, 0, 0, 0, 0, 0, 0, 0}
#define T_NOW() clock64()
#define T_ADD(i, t0) (tw_[i] += clock64() - (t0))
#define T_STAMP(i) do { if (blockIdx.x == 0) { unsigned long long t_; asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t_)); trace_words(L)[i] = t_; } } while (0)
#define T_FLUSH(lo, hi) do { if (blockIdx.x == 0) for (int i_ = (lo); i_ <= (hi); ++i_) trace_words(L)[i_] = (unsigned long long)tw_[i_]; } while (0)
#else
#define T_DECL
#define T_NOW() 0ll
#define T_ADD(i, t0) ((void)(t0))
#define T_STAMP(i) ((void)0)
#define T_FLUSH(lo, hi) ((void)0)
#define D_SPIN_LIMIT kSpinLimit
#define D_WITHHOLD_STEP -1
#endif
// One look without waiting.
__device__ __forceinline__ bool mbar_test(uint32_t bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(bar), "r"(parity)
      : "memory");
  return ok != 0;
}
// Bounded wait: false (and the wait id recorded) if the phase never completes.
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity, int* err, int id) {
  if (mbar_try_wait(bar, parity)) return true;
  const uint32_t limit = D_SPIN_LIMIT;
#pragma unroll 1
  for (uint32_t it = 0; it < limit; ++it)
    if (mbar_try_wait(bar, parity)) return true;
  atomicCAS(err, 0, id);
  return false;
}
// The same for a whole warp: every lane gets the same answer.
__device__ __forceinline__ bool warp_wait(uint32_t bar, uint32_t parity, int* err, int id) {
  return __all_sync(0xffffffffu, mbar_wait(bar, parity, err, id));
}
// Barrier `id` of `threads` threads that also tells whether `v` holds for all of them, so that a role
// in which some wait ran out leaves its loop together.
template <int ID, int THREADS>
__device__ __forceinline__ bool role_all(bool v) {
  uint32_t r;
  asm volatile(
      "{\n\t.reg .pred p, q;\n\t"
      "setp.ne.u32 q, %1, 0;\n\t"
      "bar.red.and.pred p, %2, %3, q;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(r)
      : "r"((uint32_t)v), "n"(ID), "n"(THREADS)
      : "memory");
  return r != 0;
}
// Untiled bulk copy global -> this CTA's shared memory, completing `bytes` on the mbarrier.
// Addresses 16-byte aligned, size a multiple of 16.
__device__ __forceinline__ void bulk_copy_g2s(uint32_t dst, const void* src, uint32_t bytes, uint32_t bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
               ::"r"(dst), "l"(src), "r"(bytes), "r"(bar)
               : "memory");
}
__device__ __forceinline__ void sts128(uint32_t addr, const uint32_t (&v)[4]) {
  asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(addr), "r"(v[0]), "r"(v[1]), "r"(v[2]), "r"(v[3])
               : "memory");
}
// Shared-memory matrix descriptor, K-major without swizzle: start address, distance of the two
// 8-channel halves, distance of 8-row groups, descriptor version 1.
__device__ __forceinline__ u64 smem_desc(uint32_t addr, uint32_t lbo_bytes, uint32_t sbo_bytes) {
  return (u64)((addr & 0x3FFFFu) >> 4) | ((u64)(lbo_bytes >> 4) << 16) | ((u64)(sbo_bytes >> 4) << 32) |
         (1ull << 46);
}
__device__ __forceinline__ void umma(uint32_t d_tmem, u64 a_desc, u64 b_desc, uint32_t idesc, uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}"
      ::"r"(d_tmem), "l"(a_desc), "l"(b_desc), "r"(idesc), "r"(accumulate)
      : "memory");
}
// True in exactly one lane of the (converged) warp.
__device__ __forceinline__ bool elect_one() {
  uint32_t p;
  asm volatile(
      "{\n\t.reg .pred P;\n\t"
      "elect.sync _|P, 0xFFFFFFFF;\n\t"
      "selp.u32 %0, 1, 0, P;\n\t}"
      : "=r"(p));
  return p != 0;
}
// The mbarrier receives one arrival when all MMAs issued so far by this thread have completed.
__device__ __forceinline__ void umma_commit(uint32_t bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void tmem_ld_wait() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }
__device__ __forceinline__ void tmem_ld8(uint32_t (&v)[8], uint32_t taddr) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
               : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7])
               : "r"(taddr));
}
__device__ __forceinline__ void tmem_ld16(uint32_t (&v)[16], uint32_t taddr) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
               : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]),
                 "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15])
               : "r"(taddr));
}
__device__ __forceinline__ void tmem_st8(uint32_t taddr, const float* v) {
  asm volatile("tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8};" ::"r"(taddr), "f"(v[0]), "f"(v[1]),
               "f"(v[2]), "f"(v[3]), "f"(v[4]), "f"(v[5]), "f"(v[6]), "f"(v[7])
               : "memory");
}
__device__ __forceinline__ void tmem_st_wait() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }
__device__ __forceinline__ void red_add_v4(float* p, float a, float b, float c, float d) {
  asm volatile("red.global.v4.f32.add [%0], {%1, %2, %3, %4};" ::"l"(p), "f"(a), "f"(b), "f"(c), "f"(d) : "memory");
}
// One ticket per warp: orders the warp's reductions before it and the last part's reads after it.
__device__ __forceinline__ int take_ticket(int* p) {
  int t;
  asm volatile("atom.acq_rel.gpu.global.add.s32 %0, [%1], 1;" : "=r"(t) : "l"(p) : "memory");
  return t;
}

// Work is the line of all tiles' channel steps, cut evenly among the CTAs: at tile boundaries, or (split)
// anywhere, but at least kMinSteps from one.  A CTA's share is a few segments, each inside one tile.
constexpr int kMinSteps = 2;
__host__ __device__ inline int share_begin(const DGeo& g, int cta) {
  if (g.cluster) {
    const int t = cta / g.parts;
    return t * g.k_steps + (cta - t * g.parts) * g.k_steps / g.parts;
  }
  const int x = cta * g.share + (cta < g.share_more ? cta : g.share_more);   // (tiles, or steps if split)
  if (!g.split) return x * g.k_steps;
  if (g.parts) return x;
  const int t = x / g.k_steps, r = x - t * g.k_steps;
  if (r < kMinSteps) return x - r;
  return g.k_steps - r < kMinSteps ? x - r + g.k_steps : x;
}
struct Share {
  int x0, end;
};
struct Item {
  int m0, f0, k0, k1, tile;   // first position, first filter, channel steps, number of the tile
};
// Segment s of a share; false past its last one.
__device__ __forceinline__ bool get_item(const DGeo& g, const Share& w, int s, Item* it) {
  const int x = s == 0 ? w.x0 : (w.x0 / g.k_steps + s) * g.k_steps;
  if (x >= w.end) return false;
  it->tile = x / g.k_steps;
  it->k0 = x - it->tile * g.k_steps;
  it->k1 = min(g.k_steps, it->k0 + w.end - x);
  const int mt = it->tile / g.n_ft;
  it->m0 = mt * g.mpos;
  it->f0 = (it->tile - mt * g.n_ft) * g.nt;
  return true;
}
// How many CTAs share a tile, and its part of the workspace: numbered by the first of them (no other tile
// is cut at that CTA's end), or by itself where there are fewer tiles than CTAs.
__device__ __forceinline__ void tile_owners(const DGeo& g, int tile, int* slot, int* count) {
  if (g.parts) {
    *slot = tile;
    *count = g.parts;
    return;
  }
  const int lo = tile * g.k_steps, hi = lo + g.k_steps;
  int a = max(0, lo / (g.share + 1) - 1);
  while (share_begin(g, a + 1) <= lo) ++a;
  int n = 1;
  for (int b = a + 1, x = share_begin(g, b); x < hi; ++b) {
    const int next = share_begin(g, b + 1);
    if (next > x) ++n;                                   // (a share may be empty)
    x = next;
  }
  *slot = g.n_tiles <= g.grid ? tile : a;
  *count = n;
}

// One load of the producers: V consecutive input pixels of a row (or the padding behind it).
struct Load {
  int src;    // element offset of the first pixel at channel 0, -1 = padding
  int q;      // its position inside its plane (16 bits, signed) | plane << 16 | positions it covers << 20
};
__device__ __forceinline__ Load decode_load(const DGeo& g, int m0, int u) {
  const int col = u % g.vec_cols, r = u / g.vec_cols;
  const int pa = r / g.vec_rows, row = r - pa * g.vec_rows;         // row parity plane, staged row
  const int start = m0 - g.lead;
  const int r0 = start >= 0 ? start / g.pitch : -((g.pitch - 1 - start) / g.pitch);
  const int R = r0 + row;                                           // row of the batch's line of cells
  const int e = col * g.vec;                                        // pixel of the row, in staged columns
  Load l;
  const int j = g.sx == 2 ? e >> 1 : e;
  const int cover = min(g.sx == 2 ? (g.vec + 1) >> 1 : g.vec, g.pitch - j);     // (padding ends with the row)
  l.q = ((R * g.pitch - start + j) & 0xFFFF) | (g.sx == 2 ? 2 * pa + (e & 1) : pa) << 16 | cover << 20;
  l.src = -1;
  if (R >= 0) {
    const int cell = R / g.cell_rows, i = R - cell * g.cell_rows;
    const int img = cell / g.strips, st = cell - img * g.strips;
    const int y = g.sy * i + pa, x = g.sx * (st * g.strip_w - g.ox) + e;
    if (cell < g.n_cells && y < g.h && x >= 0 && x < g.w) l.src = (img * g.c_in * g.h + y) * g.w + x;
  }
  return l;
}

// 32-bit registers of one load.
template <bool HALF, int V>
struct LoadWords { static constexpr int value = HALF ? (V + 1) / 2 : V; };
// What padding is loaded from.
__device__ uint4 g_zeros;
template <bool HALF, int V>
__device__ __forceinline__ void load_pixels(uint32_t (&v)[LoadWords<HALF, V>::value], const char* p) {
  if constexpr (LoadWords<HALF, V>::value == 2)
    asm volatile("ld.global.nc.v2.b32 {%0, %1}, [%2];" : "=r"(v[0]), "=r"(v[1]) : "l"(p));
  else if constexpr (HALF && V == 1)
    asm volatile("ld.global.nc.u16 %0, [%1];" : "=r"(v[0]) : "l"(p));
  else
    asm volatile("ld.global.nc.b32 %0, [%1];" : "=r"(v[0]) : "l"(p));
}
// {bf16(a), bf16(b)}, rounded to nearest even, a in the low half.
__device__ __forceinline__ uint32_t bf16_pair(float a, float b) {
  uint32_t r;
  asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(r) : "f"(b), "f"(a));
  return r;
}
// The same with what would round to infinity (from 3.396e38 on) as the largest finite value.
__device__ __forceinline__ uint32_t bf16_pair_sat(float a, float b) {
  uint32_t r;
  asm("cvt.rn.satfinite.bf16x2.f32 %0, %1, %2;" : "=r"(r) : "f"(b), "f"(a));
  return r;
}
// Two fp32 values as three bf16 pairs: a piece is the rest rounded to bf16, the next rest is exact, and the
// third piece holds what is left: exactly for magnitudes from 2^-110 up to the largest fp32 value, below that
// to the last bit of bf16's subnormals (2^-133).  The pieces of an infinity or a NaN add up to it again.
__device__ __forceinline__ void split_pair(float a, float b, uint32_t& p1, uint32_t& p2, uint32_t& p3) {
  p1 = bf16_pair_sat(a, b);
  a -= __uint_as_float(p1 << 16);
  b -= __uint_as_float(p1 & 0xFFFF0000u);
  p2 = bf16_pair_sat(a, b);
  a -= __uint_as_float(p2 << 16);
  b -= __uint_as_float(p2 & 0xFFFF0000u);
  p3 = bf16_pair(a, b);
}
// Eight channels of one position -> its 16-byte row(s): `v` = the channels' loads, e = which pixel of them.
// fp32: three rows, one per piece.
template <bool HALF, int V>
__device__ __forceinline__ void store_position(uint32_t dst, uint32_t slab, const uint32_t (&v)[8][LoadWords<HALF, V>::value],
                                               int e) {
  uint32_t p1[4], p2[4], p3[4];
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    if constexpr (HALF) {
      p1[i] = __byte_perm(v[2 * i][e / 2], v[2 * i + 1][e / 2], (e & 1) ? 0x7632 : 0x5410);
    } else {
      split_pair(__uint_as_float(v[2 * i][e]), __uint_as_float(v[2 * i + 1][e]), p1[i], p2[i], p3[i]);
    }
  }
  sts128(dst, p1);
  if constexpr (!HALF) {
    sts128(dst + slab, p2);
    sts128(dst + 2 * slab, p3);
  }
}

// p / d for 0 <= p < 2^31 and d >= 2 (a division by a run-time number is some 150 cycles, and a lane's
// position takes two a tile): with 2^(l-1) < d <= 2^l and mul = floor(2^(31+l) / d) + 1, mul * d exceeds
// 2^(31+l) by at most 2^l, too little to reach the next quotient.
__device__ __forceinline__ int fast_div(int p, uint32_t mul, int shift) { return (int)(__umulhi((uint32_t)p, mul) >> shift); }
void fast_div_of(int d, uint32_t* mul, int* shift) {
  int l = 1;
  while ((1ll << l) < d) ++l;
  *mul = (uint32_t)((1ull << (31 + l)) / (unsigned)d + 1);
  *shift = l - 1;
}

// Where a lane's position goes in y: element offset of filter 0, or -1 if nothing is stored there.
__device__ __forceinline__ long long position_dest(const DGeo& g, int p) {
  const int cell = fast_div(p, g.cell_mul, g.cell_shift);
  if (cell >= g.n_cells) return -1;
  const int r = p - cell * g.cell_pos;
  const int i = fast_div(r, g.pitch_mul, g.pitch_shift), j = r - i * g.pitch;
  const int img = g.strips == 1 ? cell : cell / g.strips, st = cell - img * g.strips;
  int col = st * g.strip_w + j;
  if (j >= g.strip_w) return -1;
  if (g.pool) col >>= 1;
  if (i >= g.h_out || col >= g.w_out) return -1;
  if (g.out_p8) {   // the next layer's position rows: plane and position
    const int pl = (g.out_sy == 2 ? i & 1 : 0) * g.out_sx + (g.out_sx == 2 ? col & 1 : 0);
    const int ri = g.out_sy == 2 ? i >> 1 : i, cj = g.out_sx == 2 ? col >> 1 : col;
    return (long long)pl * g.out_plane_len + g.out_lead + (img * g.out_cell_rows + ri) * g.out_pitch + cj;
  }
  return (long long)img * g.c_out * g.h_out * g.w_out + (long long)i * g.w_out + col;
}

// Eight consecutive filters f0.. of this lane's position to y: `dst` = element offset of the tile's
// first filter there (or -1), `c` = this chunk's first filter inside the tile, n_f = filters the tile
// really has.  With a fused pool the two lanes of a pair hold the same maximum: the even lane stores
// the even filters, the odd lane the odd ones.
__device__ __forceinline__ void store_chunk(float* __restrict__ y, const float (&v)[8], long long dst, int c, int n_f,
                                            size_t plane, bool pool, bool, int lane) {
  if (dst < 0) return;
  float* p = y + dst + (size_t)c * plane;
  const int room = n_f - c;
  if (pool) {
    const bool odd = lane & 1;
    if (odd) p += plane;
#pragma unroll
    for (int i = 0; i < 8; i += 2, p += 2 * plane)
      if (i + (lane & 1) < room) *p = odd ? v[i + 1] : v[i];
  } else if (room >= 8) {
#pragma unroll
    for (int i = 0; i < 8; ++i, p += plane) *p = v[i];
  } else {
#pragma unroll
    for (int i = 0; i < 8; ++i, p += plane)
      if (i < room) *p = v[i];
  }
}
// fp16: where rows are an even number of columns, the two lanes of a pair exchange a value so that
// each stores both columns of one filter (4 bytes).
__device__ __forceinline__ void store_chunk(__half* __restrict__ y, const float (&v)[8], long long dst, int c, int n_f,
                                            size_t plane, bool pool, bool pairs, int lane) {
  const int odd = lane & 1, room = n_f - c;
  __half2 own[4];                                            // filters i, i + 1 at this lane's position
#pragma unroll
  for (int i = 0; i < 4; ++i) own[i] = __floats2half2_rn(v[2 * i], v[2 * i + 1]);
  if (pool) {
    if (dst < 0) return;
    __half* p = y + dst + (size_t)(c + odd) * plane;
#pragma unroll
    for (int i = 0; i < 8; i += 2, p += 2 * plane)
      if (i + odd < room) *p = odd ? __high2half(own[i / 2]) : __low2half(own[i / 2]);
  } else if (pairs) {
    uint32_t w[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const uint32_t o = *reinterpret_cast<const uint32_t*>(&own[i]);
      const uint32_t got = __shfl_xor_sync(0xffffffffu, o, 1);
      // even lane: filter i of columns (own, next); odd lane: filter i + 1 of columns (previous, own)
      w[i] = odd ? __byte_perm(got, o, 0x7632) : __byte_perm(o, got, 0x5410);
    }
    if (dst < 0) return;
    __half* p = y + dst - odd + (size_t)(c + odd) * plane;
    if (room >= 8) {
#pragma unroll
      for (int i = 0; i < 4; ++i, p += 2 * plane) *reinterpret_cast<uint32_t*>(p) = w[i];
    } else {
#pragma unroll
      for (int i = 0; i < 4; ++i, p += 2 * plane)
        if (2 * i + odd < room) *reinterpret_cast<uint32_t*>(p) = w[i];
    }
  } else if (dst >= 0) {
    __half* p = y + dst + (size_t)c * plane;
#pragma unroll
    for (int i = 0; i < 8; ++i, p += plane)
      if (i < room) *p = i & 1 ? __high2half(own[i / 2]) : __low2half(own[i / 2]);
  }
}

// Eight consecutive filters of this lane's position as 16-byte rows of the next layer's input (`dst` =
// plane and position, `group` = the eight channels' number there); of a pooled pair the even lane stores.
template <bool HALF>
__device__ __forceinline__ void store_rows(void* __restrict__ y, const DGeo& g, const float (&v)[8], long long dst, int group,
                                           bool pool, int lane) {
  if (dst < 0 || (pool && (lane & 1))) return;
  constexpr int kPieces = HALF ? 1 : 3;
  const size_t piece = (size_t)(g.out_sy * g.out_sx) * g.out_plane_len;
  uint4* p = reinterpret_cast<uint4*>(y) + (size_t)group * kPieces * piece + dst;
  uint32_t p1[4], p2[4], p3[4];
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    float a = v[2 * i], b = v[2 * i + 1];
    if constexpr (HALF) {
      const __half2 h = __floats2half2_rn(a, b);
      p1[i] = *reinterpret_cast<const uint32_t*>(&h);
    } else {
      split_pair(a, b, p1[i], p2[i], p3[i]);
    }
  }
  p[0] = make_uint4(p1[0], p1[1], p1[2], p1[3]);
  if constexpr (!HALF) {
    p[piece] = make_uint4(p2[0], p2[1], p2[2], p2[3]);
    p[2 * piece] = make_uint4(p3[0], p3[1], p3[2], p3[3]);
  }
}

// Bias and ReLU of eight finished columns.
__device__ __forceinline__ void add_bias(float (&v)[8], const float* bias, bool relu) {
  const float4 a = reinterpret_cast<const float4*>(bias)[0], b = reinterpret_cast<const float4*>(bias)[1];
  v[0] += a.x; v[1] += a.y; v[2] += a.z; v[3] += a.w;
  v[4] += b.x; v[5] += b.y; v[6] += b.z; v[7] += b.w;
#pragma unroll
  for (int i = 0; i < 8; ++i)
    if (relu) v[i] = fmaxf(v[i], 0.f);
}
// ... and their store (filters f0 + col ..) at this lane's position, as position rows or NCHW (kEither: as
// the launch says).
enum Form { kNchw, kRows, kEither };
template <bool HALF, Form FORM>
__device__ __forceinline__ void finish_columns(const DGeo& g, void* __restrict__ y, float (&v)[8], const float* bias_s,
                                               long long dst, int f0, int col, int n_f, size_t plane, bool pool,
                                               bool pairs, int lane) {
  typedef typename std::conditional<HALF, __half, float>::type T;
  add_bias(v, bias_s + col, g.relu);
  if (FORM == kRows || (FORM == kEither && g.out_p8)) {
    // (the last filter tile may reach past the layer's filters, and so past the next layer's groups)
    if (f0 + col < g.rows) store_rows<HALF>(y, g, v, dst, (f0 + col) >> 3, pool, lane);
  } else {
    store_chunk(reinterpret_cast<T*>(y), v, dst, col, n_f, plane, pool, pairs, lane);
  }
}
// Where a lane's position goes: element offset at filter f0, or plane and position; -1: nowhere.
__device__ __forceinline__ long long lane_dest(const DGeo& g, int p, int f0, size_t plane) {
  const long long d = position_dest(g, p);
  return g.out_p8 || d < 0 ? d : d + (long long)f0 * (long long)plane;
}
// With a fused pool two tiles are the two rows of the same positions, the two lanes of a pair the two
// columns.
__device__ __forceinline__ void pool_columns(float (&v)[8], const float (&v2)[8]) {
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    v[i] = fmaxf(v[i], v2[i]);
    v[i] = fmaxf(v[i], __shfl_xor_sync(0xffffffffu, v[i], 1));
  }
}

// ---- sums that are not finite --------------------------------------------------------------------
// The dense sums hold a product for every pruned weight's zero too, and 0 x infinity is not a number; and sums of
// pieces can leave the range where the result does not.  Every output with such a term has a sum that is
// not finite.  A warp that stores one remembers the segment and, once all its work is done, forms the
// segment's outputs again from the layer's lists, over the surviving taps alone: an infinity or a NaN reaches
// the outputs that depend on it and no others.  The usual case pays four packed multiply-adds per eight columns.
// What it costs: VGG-16 N=1 331 -> 334 us, ResNet-50 N=32 855 -> 863, CIFAR VGG-16 fp16 N=256 333 -> 334.5, one
// layer 11.9 -> 12.0.  Formed again inside the epilogue loop it cost 2-6 % (registers kept for the call in all
// roles); fp32, whose epilogue has no register left for the segments, keeps them in shared memory and forms them
// at the very end, fp16 (0.5 % the other way round) in a register until the epilogue ends.
__device__ __forceinline__ void note_finite(u64& z, const uint32_t (&v)[8]) {   // two sums that stay 0 while all are finite
#pragma unroll
  for (int i = 0; i < 8; i += 2)
    asm("{\n\t.reg .b64 a, o;\n\tmov.b64 a, {%1, %2};\n\tmov.b64 o, 0;\n\tfma.rn.f32x2 %0, a, o, %0;\n\t}"
        : "+l"(z) : "r"(v[i]), "r"(v[i + 1]));
}
__device__ __forceinline__ bool all_finite(u64 z) {
  return __uint_as_float((uint32_t)z) + __uint_as_float((uint32_t)(z >> 32)) == 0.f;
}
// The bit of a segment in the warp's memory: whole tiles share 14 (all of them are this CTA's to store again);
// parts of a tile, which another CTA may have stored, can only be the share's first segment and its last.
__device__ __forceinline__ uint32_t redo_bit(const DGeo& g, const Item& it, int seg) {
  return it.k1 - it.k0 == g.k_steps ? 4u << (seg % 14) : seg == 0 ? 1u : 2u;
}

// The sum of filter o at position p of tile j.  Its input pixels are found as the staging found them: in x, or
// in the position rows behind the tap's shift.
template <bool HALF, bool P8>
__device__ __forceinline__ float sum_from_lists(const DeviceLayer& L, const DGeo& g, const void* __restrict__ xv, int p, int j,
                                                int o) {
  constexpr int kPieces = HALF ? 1 : 3;
  const int cell = p / g.cell_pos, r = p - cell * g.cell_pos, i = r / g.pitch;
  const int img = cell / g.strips, st = cell - img * g.strips;
  const int y0 = (g.pool ? 2 * i + (j & 1) : i) * L.stride - 1;
  const int x0 = (st * g.strip_w + r - i * g.pitch) * L.stride - 1;
  const size_t piece = (size_t)g.planes * g.in_plane_len * 8;          // values of one piece of eight channels
  const int end = L.row_ptr[o + 1];
  float sum = 0.f;
#pragma unroll 1
  for (int k = L.row_ptr[o]; k < end; ++k) {
    const uint32_t idx = L.csr_idx[k];
    const int c = idx & 0xFFFF;
    uint32_t mask = idx >> 16;                                         // (four taps)
#pragma unroll
    for (int s = 0; s < 4; ++s, mask &= mask - 1) {
      const int t = __ffs(mask) - 1;
      float v = 0.f;
      if constexpr (P8) {
        const int off = g.tap_off[j][__popc(L.tap_mask & ((1 << t) - 1))] - 128 * (g.pool ? j >> 1 : j);
        const int pl = off / g.plane_pos, q = g.in_lead + p + off - pl * g.plane_pos - g.lead;
        const size_t at = (size_t)(c >> 3) * kPieces * piece + ((size_t)pl * g.in_plane_len + q) * 8 + (c & 7);
        if constexpr (HALF) {
          v = __half2float(reinterpret_cast<const __half*>(xv)[at]);
        } else {
          const unsigned short* b = reinterpret_cast<const unsigned short*>(xv) + at;
          v = __uint_as_float((uint32_t)b[0] << 16) + __uint_as_float((uint32_t)b[piece] << 16) +
              __uint_as_float((uint32_t)b[2 * piece] << 16);
        }
      } else {
        const int y = y0 + t / 3, x = x0 + t % 3;
        if ((unsigned)y < (unsigned)g.h && (unsigned)x < (unsigned)g.w) {
          const size_t at = (((size_t)img * g.c_in + c) * g.h + y) * g.w + x;
          if constexpr (HALF) v = __half2float(reinterpret_cast<const __half*>(xv)[at]);
          else v = reinterpret_cast<const float*>(xv)[at];
        }
      }
      sum = fmaf(L.csr_val[4 * (size_t)k + s], v, sum);
    }
  }
  return sum;
}

// The segments of `redo` again: this warp's blocks of eight columns first, first + step, ...
template <bool HALF, bool P8>
__device__ __noinline__ void emit_from_lists(const DeviceLayer& L, const DGeo& g, uint32_t redo, const void* __restrict__ xv,
                                             const float* __restrict__ bias, void* __restrict__ yv, int first, int step) {
  typedef typename std::conditional<HALF, __half, float>::type T;
  const size_t plane = (size_t)g.h_out * g.w_out;
  const bool pool = g.pool != 0, pairs = !pool && (g.w_out & 1) == 0 && (g.strip_w & 1) == 0;
  const Share share = {share_begin(g, blockIdx.x), share_begin(g, blockIdx.x + 1)};
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int q = warp & 3, n_col = g.nt / 2, col0 = (warp >> 2) * n_col, blocks = n_col / 8, jstep = pool ? 2 : 1;
  Item it;
#pragma unroll 1
  for (int seg = 0; get_item(g, share, seg, &it); ++seg) {
    if (!(redo & redo_bit(g, it, seg))) continue;
    const int top = min(min(g.nt, g.c_out - it.f0), col0 + n_col);
#pragma unroll 1
    for (int i = first; i < g.tiles / jstep * blocks; i += step) {
      const int jj = i / blocks, col = col0 + (i - jj * blocks) * 8;
      const int p = it.m0 + 128 * jj + 32 * q + lane;
      const long long dst = lane_dest(g, p, it.f0, plane);
      float v[8];
#pragma unroll 1
      for (int k = 0; k < 8; ++k) {
        const int o = it.f0 + col + k;
        const bool real = dst >= 0 && col + k < top;
        float best = 0.f;
#pragma unroll 1
        for (int j = jstep * jj; j < jstep * jj + jstep; ++j) {
          float sum = real ? sum_from_lists<HALF, P8>(L, g, xv, p, j, o) + (bias ? bias[o] : 0.f) : 0.f;
          if (g.relu) sum = fmaxf(sum, 0.f);
          best = j == jstep * jj ? sum : fmaxf(best, sum);
        }
        v[k] = pool ? fmaxf(best, __shfl_xor_sync(0xffffffffu, best, 1)) : best;
      }
      if (g.out_p8) {
        if (it.f0 + col < g.rows) store_rows<HALF>(yv, g, v, dst, (it.f0 + col) >> 3, pool, lane);
      } else {
        store_chunk(reinterpret_cast<T*>(yv), v, dst, col, top, plane, pool, pairs, lane);
      }
    }
  }
}

// A warp's finished columns of one tile (n_col of them, the ones that are stored) from Tensor Memory to the
// result; false if a sum was not finite.
template <bool HALF, Form FORM>
__device__ __forceinline__ bool emit_columns(const DGeo& g, void* __restrict__ y, uint32_t from, uint32_t tile_stride,
                                             const float* bias_s, long long dst, int f0, int col0, int n_col, int n_f,
                                             size_t plane, bool pool, bool pairs, int lane) {
  constexpr int kWide = HALF && FORM == kNchw ? 8 : 16;
  u64 z = 0;
#pragma unroll 1
  for (int c = 0; c < n_col; c += kWide) {
    uint32_t r[kWide / 8][8];
#pragma unroll
    for (int k = 0; k < kWide / 8; ++k)
      if (c + 8 * k < n_col) tmem_ld8(r[k], from + (uint32_t)(c + 8 * k));
    tmem_ld_wait();
#pragma unroll
    for (int k = 0; k < kWide / 8; ++k) {
      if (c + 8 * k >= n_col) break;
      float v[8];
#pragma unroll
      for (int i = 0; i < 8; ++i) v[i] = __uint_as_float(r[k][i]);
      note_finite(z, r[k]);
      if (pool) {
        uint32_t r2[8];
        float v2[8];
        tmem_ld8(r2, from + tile_stride + (uint32_t)(c + 8 * k));
        tmem_ld_wait();
#pragma unroll
        for (int i = 0; i < 8; ++i) v2[i] = __uint_as_float(r2[i]);
        note_finite(z, r2);
        pool_columns(v, v2);
      }
      // (a warp stores its own columns only)
      finish_columns<HALF, FORM>(g, y, v, bias_s, dst, f0, col0 + c + 8 * k, min(n_f, col0 + n_col), plane, pool, pairs,
                                 lane);
    }
  }
  return !__any_sync(0xffffffffu, dst >= 0 && !all_finite(z));
}

// All threads of a cluster's CTAs meet; writes before it are seen after it.
__device__ __forceinline__ void cluster_sync() {
  asm volatile("barrier.cluster.arrive.release;\n\tbarrier.cluster.wait.acquire;" ::: "memory");
}
__device__ __forceinline__ float4 ld_cluster(uint32_t addr, uint32_t rank) {
  float4 v;
  asm volatile(
      "{\n\t.reg .b32 a;\n\tmapa.shared::cluster.u32 a, %4, %5;\n\t"
      "ld.shared::cluster.v4.f32 {%0, %1, %2, %3}, [a];\n\t}"
      : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w)
      : "r"(addr), "r"(rank)
      : "memory");
  return v;
}
// Sums of a warp's columns for the other CTAs of the cluster: [column / 4][warp][lane][4] fp32.
__device__ __forceinline__ uint32_t exchange_addr(uint32_t base, int c4, int warp, int lane) {
  return base + (uint32_t)((c4 * 8 + warp) * 32 + lane) * 16u;
}

// Warp roles share these shared-memory addresses.
struct Bars {
  uint32_t af, ae, bf, be, cf, ce;    // activations, weights, accumulators: full / empty
};

// ======================================= MMA issuer =======================================
// The whole warp runs this, one elected lane issues.  The tensor core takes an instruction only when it
// can start it, so every cycle of issue that is not hidden is lost, and what keeps the issue short was
// measured (128 x 128 x 16, 64 cycles each): addresses that the compiler can prove uniform (140 cycles an
// MMA otherwise), tile count and product schedule known at compile time (a tap with a run-time tile loop:
// 630 cycles instead of 390), and a wait whose usual case is one try without any state carried across
// (+40 cycles a tap otherwise).
template <bool HALF, bool P8, int TILES, bool FORM3>
__device__ __forceinline__ void mma_role(const DeviceLayer& L, const DGeo& g, uint32_t sbase, uint32_t tmem, const Bars& bar,
                                         const Share& share, int lane) {
  using C = Cfg<HALF, P8>;
  // One MMA.  (Electing for each one leaves the address arithmetic outside the elected region, where it can
  // use the uniform pipeline.)
  auto mma = [&](uint32_t d, u64 a, u64 b, uint32_t idesc, uint32_t acc) {
    if (elect_one()) umma(d, a, b, idesc, acc);
  };
    const uint32_t id0 = (1u << 4) | (HALF ? 0u : (1u << 7) | (1u << 10)) | ((128u >> 4) << 24);
    const uint32_t nt = (uint32_t)g.nt;
    const uint32_t id1 = id0 | ((nt >> 3) << 17), id2 = id0 | ((2 * nt >> 3) << 17), id3 = id0 | ((3 * nt >> 3) << 17);
    // (in a cluster a shared-memory address carries the CTA's rank above its 18 bits; descriptors do not)
    const uint32_t sdesc = sbase & 0x3FFFFu;
    const u64 a_d0 = smem_desc(0u, (uint32_t)g.q_tot * 16u, 128u);
    const u64 b_d0 = smem_desc(0u, (uint32_t)(C::kPieces * g.nt) * 16u, 128u);
    const uint32_t slab = 2u * (uint32_t)g.q_tot;        // 16-byte rows of one piece of a stage
    const uint32_t tap_rows = (uint32_t)(2 * C::kPieces * g.nt);
    int sa = 0, pa = 0, sb = 0, pb = 0;
    uint32_t sc = 0;                                     // fp32: channel steps so far; fp16: items
    bool failed = false;
    T_DECL;
    const long long t_all = T_NOW();
    // After a wait that ran out nothing is waited for any more; the loops go on, so that their control
    // flow -- and with it every address -- stays visibly uniform, and the other roles get their signals.
    auto wait = [&](uint32_t b, int parity, int id, int trace) {
      const long long t_ = T_NOW();
      if (!mbar_test(b, (uint32_t)parity))
        if (!failed) failed = !warp_wait(b, (uint32_t)parity, L.err, id);
      T_ADD(trace, t_);
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    };
    auto slot_desc = [&](int s) -> u64 {
      return b_d0 + ((sdesc + (uint32_t)g.b_off + (uint32_t)s * (uint32_t)g.b_bytes) >> 4);
    };
    Item it;
    for (int seg = 0; get_item(g, share, seg, &it); ++seg) {
      if constexpr (HALF) {
        const uint32_t buf = g.n_buf == 2 ? (sc & 1u) : 0u, use = g.n_buf == 2 ? sc >> 1 : sc;
        wait(bar.ce + 8 * buf, (use & 1u) ^ 1u, kWaitSums, 1);
        const uint32_t d0 = tmem + buf * 256u;
        for (int ks = it.k0; ks < it.k1; ++ks) {
          wait(bar.af + 8 * sa, pa, kWaitFull, 2);
          const u64 a_st = a_d0 + ((sdesc + (uint32_t)g.a_off + (uint32_t)sa * (uint32_t)g.a_bytes) >> 4);
#pragma unroll
          for (int t = 0; t < 9; t += 3) {                 // three taps to a slot
            if (t >= g.n_taps) break;
            wait(bar.bf + 8 * sb, pb, kWaitFull, 3);
            const u64 b_t = slot_desc(sb);
#pragma unroll
            for (int v = 0; v < 3; ++v) {
              if (t + v >= g.n_taps) break;
              const uint32_t acc = (ks > it.k0 || t + v > 0) ? 1u : 0u;
#pragma unroll
              for (int j = 0; j < TILES; ++j)
                mma(d0 + (uint32_t)(j * g.tile_cols), a_st + (uint32_t)g.tap_off[j][t + v],
                    b_t + (uint32_t)v * tap_rows, id1, acc);
            }
            if (elect_one()) umma_commit(bar.be + 8 * sb);
            if (++sb == g.b_slots) { sb = 0; pb ^= 1; }
          }
          if (elect_one()) umma_commit(bar.ae + 8 * sa);
          if (++sa == g.a_stages) { sa = 0; pa ^= 1; }
        }
        if (elect_one()) umma_commit(bar.cf + 8 * buf);    // the item's accumulators are complete
        ++sc;
      } else {
        // Cross products of the first two taps, then -- once the epilogue warps have taken the main sums
        // of the last step -- their main products, then the other taps.
        for (int ks = it.k0; ks < it.k1; ++ks, ++sc) {
          const bool first = ks == it.k0;
          if (first) wait(bar.ce, (sc & 1u) ^ 1u, kWaitSums, 1);
          wait(bar.af + 8 * sa, pa, kWaitFull, 2);
          const u64 a_st = a_d0 + ((sdesc + (uint32_t)g.a_off + (uint32_t)sa * (uint32_t)g.a_bytes) >> 4);
          auto cross = [&](int j, int t, u64 b_t) {
            const u64 a1 = a_st + (uint32_t)g.tap_off[j][t], a2 = a1 + slab, a3 = a2 + slab;
            const uint32_t dc = tmem + (uint32_t)(j * g.tile_cols) + nt;
            const uint32_t acc = (!first || t > 0) ? 1u : 0u;
            if constexpr (FORM3) {       // columns main | cross | second cross
              mma(dc, a2, b_t, id2, acc);
              mma(dc, a3, b_t, id1, 1u);
            } else {             // columns main | cross
              mma(dc, a2, b_t, id1, acc);
              mma(dc, a2, b_t + nt, id1, 1u);
              mma(dc, a3, b_t, id1, 1u);
              mma(dc, a1, b_t + 2 * nt, id1, 1u);
            }
          };
          auto main = [&](int j, int t, u64 b_t) {
            const u64 a1 = a_st + (uint32_t)g.tap_off[j][t];
            const uint32_t dm = tmem + (uint32_t)(j * g.tile_cols);
            if (t == 0) {        // the main sums start afresh in every step, the cross sums go on
              mma(dm, a1, b_t, id1, 0u);
              mma(dm + nt, a1, b_t + nt, FORM3 ? id2 : id1, 1u);
            } else {
              mma(dm, a1, b_t, FORM3 ? id3 : id2, 1u);
            }
          };
          constexpr int kPre = 5;
          int s2 = sb, p2 = pb;
#pragma unroll
          for (int t = 0; t < kPre; ++t) {
            if (t >= g.n_taps) break;
            wait(bar.bf + 8 * s2, p2, kWaitFull, 3);
            const u64 b_t = slot_desc(s2);
#pragma unroll
            for (int j = 0; j < TILES; ++j) cross(j, t, b_t);
            if (++s2 == g.b_slots) { s2 = 0; p2 ^= 1; }
          }
          if (!first) wait(bar.ce, (sc & 1u) ^ 1u, kWaitSums, 1);
#pragma unroll
          for (int t = 0; t < 9; ++t) {
            if (t >= g.n_taps) break;
            if (t >= kPre) wait(bar.bf + 8 * sb, pb, kWaitFull, 3);
            const u64 b_t = slot_desc(sb);
#pragma unroll
            for (int j = 0; j < TILES; ++j) {
              if (t >= kPre) cross(j, t, b_t);
              main(j, t, b_t);
            }
            if (elect_one()) umma_commit(bar.be + 8 * sb);
            if (++sb == g.b_slots) { sb = 0; pb ^= 1; }
          }
          if (elect_one()) {
            umma_commit(bar.cf);
            umma_commit(bar.ae + 8 * sa);
          }
          if (++sa == g.a_stages) { sa = 0; pa ^= 1; }
        }
      }
    }
    T_ADD(0, t_all);
    if (lane == 0) T_FLUSH(0, 3);
}

// ======================================= weight stream ====================================
// Per slot six bulk copies (or one, where a slot is one run).  Written like the MMA issuer, with uniform
// addresses and control flow: one elected lane looping over the copies took ~60 cycles for each and could
// not keep up with the MMAs.  Weights do not depend on the previous kernel of the stream: no wait for it.
template <bool HALF>
__device__ __forceinline__ void weight_role(const DeviceLayer& L, const DGeo& g, uint32_t sbase, const Bars& bar,
                                            const Share& share, int lane) {
  constexpr int kTapRuns = 2 * (HALF ? 1 : 3), kTps = HALF ? 3 : 1;
  const size_t row_b = (size_t)g.rows * 16;                   // one (8 channels, piece) run of all filters
  const char* wd = reinterpret_cast<const char*>(L.wdense);
  const bool whole = g.rows == g.nt;                          // one filter tile: a slot is one run
  int sb = 0, pb = 0;
  bool failed = false, wrapped = false;
  T_DECL;
  Item it;
  for (int seg = 0; get_item(g, share, seg, &it); ++seg) {
    const int rows = min(g.nt, g.rows - it.f0);               // the last filter tile may be short
    const uint32_t run = (uint32_t)rows * 16u, run_s = (uint32_t)g.nt * 16u;
    for (int ks = it.k0; ks < it.k1; ++ks) {
      const char* src = wd + (size_t)ks * g.n_taps * kTapRuns * row_b + (size_t)it.f0 * 16;
      for (int t = 0; t < g.n_taps; t += kTps) {
        const int runs = min(kTps, g.n_taps - t) * kTapRuns;
        const uint32_t slot_bar = bar.bf + 8 * sb;
        const long long t_ = T_NOW();
        if (!mbar_test(bar.be + 8 * sb, (uint32_t)(pb ^ 1)))
          if (!failed) failed = !warp_wait(bar.be + 8 * sb, (uint32_t)(pb ^ 1), L.err, kWaitFree);
        T_ADD(6, t_);
        const uint32_t dst = sbase + (uint32_t)g.b_off + (uint32_t)sb * (uint32_t)g.b_bytes;
        if (failed) break;
        if (whole) {
          if (elect_one()) {
            mbar_arrive_expect_tx(slot_bar, (uint32_t)runs * run_s);
            bulk_copy_g2s(dst, src, (uint32_t)runs * run_s, slot_bar);
          }
        } else {
          if (elect_one()) mbar_arrive_expect_tx(slot_bar, (uint32_t)runs * run);
#pragma unroll
          for (int r = 0; r < kTps * kTapRuns; ++r)
            if (r < runs && elect_one()) bulk_copy_g2s(dst + r * run_s, src + r * row_b, run, slot_bar);
        }
        src += (size_t)runs * row_b;
        if (++sb == g.b_slots) { sb = 0; pb ^= 1; wrapped = true; }
      }
      if (failed) break;
    }
    if (failed) break;
  }
  // no copy is in flight when the CTA ends, whatever made it end
  for (int s = 0; s < g.b_slots; ++s) {
    if (s >= sb && !wrapped) break;
    warp_wait(bar.bf + 8 * s, (uint32_t)(s < sb ? pb : pb ^ 1), L.err, kWaitFull);
  }
  if (lane == 0) T_FLUSH(6, 6);
}

// ======================================= activations ======================================
// Source in position rows: the slab of a step is one run of positions per (piece, 8 channels, plane), one
// bulk copy each.
template <bool HALF>
__device__ __forceinline__ void activation_role(const DeviceLayer& L, const DGeo& g, uint32_t sbase, const Bars& bar,
                                                const Share& share, const void* x, int lane) {
  constexpr int kPieces = HALF ? 1 : 3;
  const int withhold = D_WITHHOLD_STEP;     // (development build: a step that is never staged)
  const size_t plane_b = (size_t)g.in_plane_len * 16, piece_b = plane_b * g.planes;
  const uint32_t run = (uint32_t)g.plane_pos * 16u, bytes = 2u * kPieces * (uint32_t)g.planes * run;
  int sa = 0, pa = 0;
  bool failed = false, wrapped = false;
  T_DECL;
  // the previous kernel of the stream has finished before x is read
  asm volatile("griddepcontrol.wait;" ::: "memory");
  if (lane == 0) T_STAMP(11);
  Item it;
  for (int seg = 0; get_item(g, share, seg, &it); ++seg) {
    const char* xi = reinterpret_cast<const char*>(x) + (size_t)(it.m0 + g.in_lead - g.lead) * 16;
    for (int ks = it.k0; ks < it.k1; ++ks) {
      const long long t_ = T_NOW();
      if (!mbar_test(bar.ae + 8 * sa, (uint32_t)(pa ^ 1)))
        if (!failed) failed = !warp_wait(bar.ae + 8 * sa, (uint32_t)(pa ^ 1), L.err, kWaitFree);
      T_ADD(5, t_);
      if (failed || ks - it.k0 == withhold) break;
      const uint32_t full = bar.af + 8 * sa;
      if (elect_one()) mbar_arrive_expect_tx(full, bytes);
      uint32_t dst = sbase + (uint32_t)g.a_off + (uint32_t)sa * (uint32_t)g.a_bytes;
      const char* src = xi + (size_t)(2 * ks) * kPieces * piece_b;
#pragma unroll
      for (int p = 0; p < kPieces; ++p)
#pragma unroll
        for (int kh = 0; kh < 2; ++kh) {
          const char* sp = src + (size_t)(kh * kPieces + p) * piece_b;
          for (int pl = 0; pl < g.planes; ++pl, dst += run, sp += plane_b)
            if (elect_one()) bulk_copy_g2s(dst, sp, run, full);
        }
      if (++sa == g.a_stages) { sa = 0; pa ^= 1; wrapped = true; }
    }
    if (failed) break;
  }
  // no copy is in flight when the CTA ends, whatever made it end
  for (int s = 0; s < g.a_stages; ++s) {
    if (s >= sa && !wrapped) break;
    warp_wait(bar.af + 8 * s, (uint32_t)(s < sa ? pa : pa ^ 1), L.err, kWaitFull);
  }
  if (lane == 0) T_FLUSH(5, 5);
}

template <bool HALF, int V>
__global__ void __launch_bounds__(Cfg<HALF, V == 0>::kThreads, 1)
dense_kernel(const __grid_constant__ DeviceLayer L, const __grid_constant__ DGeo g, const void* __restrict__ xv,
             const float* __restrict__ bias, void* __restrict__ yv, float* __restrict__ ws, int* __restrict__ tickets) {
  constexpr bool P8 = V == 0;
  using C = Cfg<HALF, P8>;
  extern __shared__ __align__(1024) unsigned char smem[];
  const uint32_t sbase = smem_u32(smem);
  const int tid = threadIdx.x, lane = tid & 31;
  const int warp = __shfl_sync(0xffffffffu, tid >> 5, 0);
  const uint32_t bar_af = sbase, bar_ae = bar_af + 8 * kMaxA;
  const uint32_t bar_bf = bar_ae + 8 * kMaxA, bar_be = bar_bf + 8 * kMaxB;
  const uint32_t bar_cf = bar_be + 8 * kMaxB, bar_ce = bar_cf + 16;     // accumulators full / empty
  volatile uint32_t* tmem_s = reinterpret_cast<volatile uint32_t*>(smem + 16 * (kMaxA + kMaxB) + 32);
  volatile uint16_t* redo_s = reinterpret_cast<volatile uint16_t*>(tmem_s + 1);     // [8] fp32: see redo_bit
  float* bias_s = reinterpret_cast<float*>(smem + kBiasOff);            // [128]
  Load* tab_s = reinterpret_cast<Load*>(smem + kHeader);                // [kTables][n_vec]

  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  if (tid == 0) T_STAMP(10);
  if (tid == 0) {
    for (int s = 0; s < g.a_stages; ++s) {
      mbar_init(bar_af + 8 * s, C::kProdWarps);
      mbar_init(bar_ae + 8 * s, 1);
    }
    for (int s = 0; s < g.b_slots; ++s) {
      mbar_init(bar_bf + 8 * s, 1);
      mbar_init(bar_be + 8 * s, 1);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(bar_cf + 8 * b, 1);
      mbar_init(bar_ce + 8 * b, C::kEpiWarps);
    }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (!HALF && tid < C::kEpiWarps) redo_s[tid] = 0;
  if (warp == C::kMmaWarp) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 512;" ::"r"(
                     smem_u32((const void*)tmem_s))
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = __shfl_sync(0xffffffffu, *tmem_s, 0);
  const size_t hw = (size_t)g.h * g.w;
  const Bars bars = {bar_af, bar_ae, bar_bf, bar_be, bar_cf, bar_ce};
  const Share share = {share_begin(g, blockIdx.x), share_begin(g, blockIdx.x + 1)};
  if (warp == C::kMmaWarp) {
    // ======================================= MMA issuer =======================================
    if constexpr (HALF) {
      if (g.tiles == 4) mma_role<true, P8, 4, false>(L, g, sbase, tmem, bars, share, lane);
      else if (g.tiles == 2) mma_role<true, P8, 2, false>(L, g, sbase, tmem, bars, share, lane);
      else mma_role<true, P8, 1, false>(L, g, sbase, tmem, bars, share, lane);
    } else {
      if (g.tiles == 2 && g.form3) mma_role<false, P8, 2, true>(L, g, sbase, tmem, bars, share, lane);
      else if (g.tiles == 2) mma_role<false, P8, 2, false>(L, g, sbase, tmem, bars, share, lane);
      else if (g.form3) mma_role<false, P8, 1, true>(L, g, sbase, tmem, bars, share, lane);
      else mma_role<false, P8, 1, false>(L, g, sbase, tmem, bars, share, lane);
    }
    __syncwarp();
  } else if (warp == C::kBWarp) {
    weight_role<HALF>(L, g, sbase, bars, share, lane);
    __syncwarp();
  } else if (warp >= C::kProdWarp0) {
    // ======================================= activations ======================================
    if constexpr (P8) {
      activation_role<HALF>(L, g, sbase, bars, share, xv, lane);
      __syncwarp();
    } else {
    constexpr int kEs = HALF ? 2 : 4;
    const char* x = reinterpret_cast<const char*>(xv);
    const size_t chan = hw * kEs;                               // bytes between channels
    const int pt = tid - 32 * C::kProdWarp0;
    const int n_tasks = 2 * g.n_vec;                            // (8 channels, load)
    const uint32_t half_b = (uint32_t)g.q_tot * 16u, slab = 2u * half_b;
    const int withhold = D_WITHHOLD_STEP;     // (development build: a step whose first warp never reports)
    T_DECL;
    // The loads of a segment: worked out three segments ahead of the stores.  A segment may be as short as
    // one batch, and two batches beyond the one to be stored next are loaded before its segment begins.
    auto fill_table = [&](int seg) {
      Item it;
      if (!get_item(g, share, seg, &it)) return;
      Load* tab = tab_s + (seg % kTables) * g.n_vec;
      for (int u = pt; u < g.n_vec; u += C::kProdThreads) tab[u] = decode_load(g, it.m0, u);
    };
    for (int i = 0; i < 3; ++i) fill_table(i);
    bool ok = role_all<1, C::kProdThreads>(true);
    // the previous kernel of the stream has finished before x is read
    asm volatile("griddepcontrol.wait;" ::: "memory");
    const long long t_all = T_NOW();
    if (pt == 0) T_STAMP(11);
    // A batch is one task a thread; batches run on through steps and items.
    struct Set {
      uint32_t v[8][LoadWords<HALF, V>::value];
      int q;
    };
    int l_seg = 0, l_t = pt, l_ks = 0, l_k1 = 0;
    const Load* l_tab = nullptr;      // (null: nothing is left to load)
    auto open_item = [&]() {
      Item it;
      l_tab = nullptr;
      if (!get_item(g, share, l_seg, &it)) return;
      l_ks = it.k0;
      l_k1 = it.k1;
      l_tab = tab_s + (l_seg % kTables) * g.n_vec;
    };
    open_item();
    auto load_batch = [&](Set& r) {
      if (!l_tab) return;
      if (l_t < n_tasks) {
        const int kh = l_t >= g.n_vec ? 1 : 0;
        const Load l = l_tab[l_t - kh * g.n_vec];
        const int c0 = l_ks * 16 + kh * 8;
        // Padding, and eight channels past the last one, read zeros; a single channel past the last one
        // reads the last one again (its weights are zero).
        const int nc = g.c_in - c0;
        const bool real = l.src >= 0 && nc > 0;
        const char* p = real ? x + (size_t)l.src * kEs + (size_t)c0 * chan : reinterpret_cast<const char*>(&g_zeros);
        const size_t stride = real ? chan : 0;
        r.q = l.q;
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          load_pixels<HALF, V>(r.v[i], p);
          if (i + 1 < nc) p += stride;
        }
      }
      l_t += C::kProdThreads;
      if (l_t - pt >= n_tasks) {
        l_t = pt;
        if (++l_ks == l_k1) {
          ++l_seg;
          open_item();
        }
      }
    };
    // Store side; false when nothing is left to store.
    int s_seg = 0, s_t = pt, s_ks = -1, s_k0 = 0, s_k1 = 0, sa = 0, pa = 0;
    auto store_batch = [&](const Set& r) -> bool {
      if (s_ks < 0) {
        Item it;
        if (!get_item(g, share, s_seg, &it)) return false;
        s_ks = s_k0 = it.k0;
        s_k1 = it.k1;
        fill_table(s_seg + 3);
        ok = role_all<1, C::kProdThreads>(ok);
        if (!ok) return false;
      }
      if (s_t == pt) {
        const long long t_ = T_NOW();
        ok = ok && mbar_wait(bar_ae + 8 * sa, (uint32_t)(pa ^ 1), L.err, kWaitFree);
        T_ADD(5, t_);
      }
      if (ok && s_t < n_tasks) {
        const int q = (int)(short)r.q, plane = r.q >> 16 & 15, cover = r.q >> 20;
        const uint32_t dst = sbase + (uint32_t)g.a_off + (uint32_t)sa * (uint32_t)g.a_bytes +
                             (s_t >= g.n_vec ? half_b : 0u) + (uint32_t)(plane * g.plane_pos + q) * 16u;
#pragma unroll
        for (int e = 0; e < V; ++e) {
          // (stride 2: odd columns go to the second plane of the pair)
          const int dq = g.sx == 2 ? e >> 1 : e;
          const uint32_t off = (uint32_t)(dq + (g.sx == 2 && (e & 1) ? g.plane_pos : 0)) * 16u;
          if (dq < cover && (unsigned)(q + dq) < (unsigned)g.plane_pos)
            store_position<HALF, V>(dst + off, slab, r.v, e);
        }
      }
      s_t += C::kProdThreads;
      if (s_t - pt >= n_tasks) {
        s_t = pt;
        // generic-proxy stores must be visible to the tensor core's (async proxy) reads
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        if (!(pt < 32 && s_ks - s_k0 == withhold)) warp_arrive(bar_af + 8 * sa, lane);
        if (++sa == g.a_stages) { sa = 0; pa ^= 1; }
        if (++s_ks == s_k1) {
          s_ks = -1;
          ++s_seg;
        }
      }
      return true;
    };
    // (three sets rotated by register moves: a loop unrolled by three overflows the instruction caches,
    // and the warps then wait for instructions instead of data)
    Set v0, v1, v2;
    load_batch(v0);
    load_batch(v1);
#pragma unroll 1
    do {
      load_batch(v2);
      const Set now = v0;
      v0 = v1;
      v1 = v2;
      if (!store_batch(now)) break;
    } while (true);
    T_ADD(4, t_all);
    if (pt == 0) T_FLUSH(4, 5);
    }
  } else {
    // ======================================= epilogue =========================================
    // fp32 keeps a warp's columns of all tiles in registers: kSums of one tile or half as many of each of two
    constexpr int kSums = HALF ? 8 : (P8 ? 128 : 64), kHalf = kSums / 2;
    const int q = warp & 3, grp = warp >> 2;             // lane quadrant, column group
    const int n_col = g.nt / C::kGroups;                 // this warp's columns of every tile
    const int col0 = grp * n_col;
    const uint32_t lane_addr = tmem + ((uint32_t)(32 * q) << 16) + (uint32_t)col0;
    const size_t plane = (size_t)g.h_out * g.w_out;
    const bool pool = g.pool != 0;
    const bool pairs = !pool && (g.w_out & 1) == 0 && (g.strip_w & 1) == 0;
    uint32_t sc = 0;
    T_DECL;
    bool ok = true, waited = false;
    uint32_t redo = 0;
    Item it;
    for (int seg = 0; get_item(g, share, seg, &it); ++seg) {
      const int n_f = min(g.nt, g.c_out - it.f0);        // real filters of this tile
      if (tid < 128) bias_s[tid] = (bias && tid < n_f) ? __ldg(bias + it.f0 + tid) : 0.f;
      float sum[kSums];
      uint32_t buf = 0;
      if constexpr (HALF) {
        buf = g.n_buf == 2 ? (sc & 1u) : 0u;
        const long long t_ = T_NOW();
        ok = warp_wait(bar_cf + 8 * buf, (g.n_buf == 2 ? sc >> 1 : sc) & 1u, L.err, kWaitSums);
        T_ADD(7, t_);
        ++sc;
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      } else {
        // adds the columns at `off` of every tile
        auto take = [&](int off) {
          // (16 columns at a time; where n_col is an odd multiple of 8 the last eight are a neighbour's)
#pragma unroll
          for (int k = 0; k < kSums; k += 16) {
            const int j = g.tiles == 2 ? k / kHalf : 0, c = g.tiles == 2 ? k % kHalf : k;
            if (c < n_col) {
              uint32_t v[16];
              tmem_ld16(v, lane_addr + (uint32_t)(j * g.tile_cols + off + c));
              tmem_ld_wait();
#pragma unroll
              for (int i = 0; i < 16; ++i) sum[k + i] += __uint_as_float(v[i]);
            }
          }
        };
#pragma unroll
        for (int k = 0; k < kSums; ++k) sum[k] = 0.f;
        // main sums of every channel step: Tensor Memory -> fp32 registers
        for (int ks = it.k0; ks < it.k1 && ok; ++ks, ++sc) {
          const long long t_ = T_NOW();
          ok = warp_wait(bar_cf, sc & 1u, L.err, kWaitSums);
          T_ADD(7, t_);
          asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
          const long long t_main = T_NOW();
          take(0);
          T_ADD(8, t_main);
          // (after the last step the cross sums are still to be read)
          if (ks + 1 < it.k1) {
            asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
            warp_arrive(bar_ce, lane);
          }
        }
        if (ok) {
          take(g.nt);
          if (g.form3) take(2 * g.nt);
        }
        // The sums go back to Tensor Memory, which can be addressed at run time: what follows is then one short
        // loop over columns.  (Unrolled over registers it was 38 KB of code run once per tile, and fetching
        // the instructions took 10 us.)  Where all columns are in use they replace the main sums.
#pragma unroll
        for (int k = 0; k < kSums; k += 8) {
          const int j = g.tiles == 2 ? k / kHalf : 0, c = g.tiles == 2 ? k % kHalf : k;
          if (c < n_col) tmem_st8(lane_addr + (uint32_t)(g.out_col + j * g.out_stride + c), sum + k);
        }
        tmem_st_wait();
        if (g.out_col) {
          asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
          warp_arrive(bar_ce, lane);
        }
      }
      if (!waited) {   // the previous kernel of the stream has finished before y or the workspace is written
        asm volatile("griddepcontrol.wait;" ::: "memory");
        waited = true;
      }
      ok = role_all<2, 32 * C::kEpiWarps>(ok);             // the bias is staged
      if (!ok) break;
      const uint32_t res = lane_addr + (HALF ? buf * 256u : (uint32_t)g.out_col);     // this warp's columns of tile 0
      const uint32_t res_stride = (uint32_t)(HALF ? g.tile_cols : g.out_stride);
      if (g.cluster) {   // this CTA's only segment: hand the sums over (the rings are free: all MMAs are done)
        for (int j = 0; j < g.tiles; ++j)
#pragma unroll 1
          for (int c = 0; c < n_col; c += 8) {
            uint32_t v[8];
            tmem_ld8(v, res + (uint32_t)j * res_stride + (uint32_t)c);
            tmem_ld_wait();
            const int c4 = (j * n_col + c) / 4;
            const uint32_t lo[4] = {v[0], v[1], v[2], v[3]}, hi[4] = {v[4], v[5], v[6], v[7]};
            sts128(exchange_addr(sbase + (uint32_t)g.a_off, c4, warp, lane), lo);
            sts128(exchange_addr(sbase + (uint32_t)g.a_off, c4 + 1, warp, lane), hi);
          }
        continue;
      }
      // Parts of the channel range: add this part's sums to the tile's in the workspace
      // ([tile][column / 4][position][4]: 16 bytes a lane), take a ticket for this warp's share; the
      // warp that draws the last one reads the sums back (zeroing them) and finishes.
      bool finish = true;
      if (it.k1 - it.k0 < g.k_steps) {
        int slot, parts;
        tile_owners(g, it.tile, &slot, &parts);
        float* wsw = ws + ((size_t)slot * g.tiles * (g.nt / 4) + (size_t)(col0 / 4)) * 512 + (size_t)(32 * q + lane) * 4;
        for (int j = 0; j < g.tiles; ++j) {
          float* pw = wsw + (size_t)(j * (g.nt / 4)) * 512;
#pragma unroll 1
          for (int c = 0; c < n_col; c += 8, pw += 1024) {
            uint32_t v[8];
            tmem_ld8(v, res + (uint32_t)j * res_stride + (uint32_t)c);
            tmem_ld_wait();
            red_add_v4(pw, __uint_as_float(v[0]), __uint_as_float(v[1]), __uint_as_float(v[2]), __uint_as_float(v[3]));
            red_add_v4(pw + 512, __uint_as_float(v[4]), __uint_as_float(v[5]), __uint_as_float(v[6]),
                       __uint_as_float(v[7]));
          }
        }
        __syncwarp();
        int t = 0;
        int* ticket = tickets + (size_t)slot * C::kEpiWarps + warp;
        if (lane == 0) {
          t = take_ticket(ticket);
          if (t == parts - 1) *ticket = 0;
        }
        finish = __shfl_sync(0xffffffffu, t, 0) == parts - 1;
        for (int j = 0; finish && j < g.tiles; ++j)
#pragma unroll 1
          for (int c = 0; c < n_col; c += 32) {       // (eight loads in flight)
            float4* pw = reinterpret_cast<float4*>(wsw + (size_t)(j * (g.nt / 4) + c / 4) * 512);
            float v[32];
#pragma unroll
            for (int i = 0; i < 8; ++i)
              if (c + 4 * i < n_col) {
                const float4 a = __ldcg(pw + 128 * i);
                v[4 * i] = a.x; v[4 * i + 1] = a.y; v[4 * i + 2] = a.z; v[4 * i + 3] = a.w;
              }
#pragma unroll
            for (int i = 0; i < 8; ++i)
              if (c + 4 * i < n_col) pw[128 * i] = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
            for (int i = 0; i < 32; i += 8)
              if (c + i < n_col) tmem_st8(res + (uint32_t)j * res_stride + (uint32_t)(c + i), v + i);
            tmem_st_wait();
          }
      }
      const long long t_fin = T_NOW();
      if (finish) {
        // fp16: one loop for each form of the result, each as short as it can be: eight warps cannot hide much
        // of each other's latency, and these loops run beside the other roles' code in small instruction caches
        // (one loop with both forms in it took 1.2-1.4 times as long).  In the fp32 kernel, whose register sums
        // leave no room, two loops cost spills in the channel loop and a fifth of its time.
        const int jstep = pool ? 2 : 1;
        // (position rows have the padding filters too; past them a tile's columns hold whatever was there)
        const int n_stored = min(n_col, (((g.out_p8 ? g.rows - it.f0 : n_f) + 7) & ~7) - col0);
        for (int j = 0, jj = 0; j < g.tiles; j += jstep, ++jj) {
          const long long dst = lane_dest(g, it.m0 + 128 * jj + 32 * q + lane, it.f0, plane);
          const uint32_t from = res + (uint32_t)j * res_stride;
          bool fine;
          if constexpr (!HALF) fine = emit_columns<HALF, kEither>(g, yv, from, res_stride, bias_s, dst, it.f0, col0, n_stored, n_f, plane, pool, pairs, lane);
          else if (g.out_p8) fine = emit_columns<HALF, kRows>(g, yv, from, res_stride, bias_s, dst, it.f0, col0, n_stored, n_f, plane, pool, pairs, lane);
          else fine = emit_columns<HALF, kNchw>(g, yv, from, res_stride, bias_s, dst, it.f0, col0, n_stored, n_f, plane, pool, pairs, lane);
          if (!fine) {
            if (HALF) redo |= redo_bit(g, it, seg);
            else redo_s[warp] = (uint16_t)(redo_s[warp] | redo_bit(g, it, seg));
          }
        }
      }
      if (!HALF && !g.out_col) {
        asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
        warp_arrive(bar_ce, lane);
      }
      if (HALF) {
        asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
        warp_arrive(bar_ce + 8 * buf, lane);
      }
      T_ADD(9, t_fin);
      asm volatile("bar.sync 2, %0;" ::"n"(32 * C::kEpiWarps) : "memory");   // the bias may be overwritten
    }
    if (tid == 0) T_FLUSH(7, 9);
    if (tid == 0) T_STAMP(12);
    if (!waited) asm volatile("griddepcontrol.wait;" ::: "memory");
    if (HALF && redo) emit_from_lists<HALF, P8>(L, g, redo, xv, bias, yv, 0, 1);
  }

  if (g.cluster) {
    // The CTAs of a tile share out its columns: each adds up its eight-column blocks over all of them, in
    // rank order, and finishes them.
    cluster_sync();
    Item it;
    if (warp < C::kEpiWarps && get_item(g, share, 0, &it)) {
      uint32_t rank;
      asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(rank));
      const int q = warp & 3, n_col = g.nt / C::kGroups, col0 = (warp >> 2) * n_col;
      const int n_f = min(g.nt, g.c_out - it.f0);
      const size_t plane = (size_t)g.h_out * g.w_out;
      const bool pool = g.pool != 0;
      const bool pairs = !pool && (g.w_out & 1) == 0 && (g.strip_w & 1) == 0;
      const uint32_t xb = sbase + (uint32_t)g.a_off;
      auto gather = [&](int c4, float (&v)[8]) {
#pragma unroll
        for (int i = 0; i < 8; ++i) v[i] = 0.f;
#pragma unroll 1
        for (int p0 = 0; p0 < g.parts; p0 += 4) {
          float4 a[4], b[4];
#pragma unroll
          for (int p = 0; p < 4; ++p)
            if (p0 + p < g.parts) {
              a[p] = ld_cluster(exchange_addr(xb, c4, warp, lane), (uint32_t)(p0 + p));
              b[p] = ld_cluster(exchange_addr(xb, c4 + 1, warp, lane), (uint32_t)(p0 + p));
            }
#pragma unroll
          for (int p = 0; p < 4; ++p)
            if (p0 + p < g.parts) {
              v[0] += a[p].x; v[1] += a[p].y; v[2] += a[p].z; v[3] += a[p].w;
              v[4] += b[p].x; v[5] += b[p].y; v[6] += b[p].z; v[7] += b[p].w;
            }
        }
      };
      const int jstep = pool ? 2 : 1, blocks = n_col / 8;
      uint32_t redo = 0;
#pragma unroll 1
      for (int i = (int)rank; i < g.tiles / jstep * blocks; i += g.parts) {
        const int jj = i / blocks, c = (i - jj * blocks) * 8;
        const long long dst = lane_dest(g, it.m0 + 128 * jj + 32 * q + lane, it.f0, plane);
        float v[8], v2[8], z = 0.f;
        gather((jj * jstep * n_col + c) / 4, v);
#pragma unroll
        for (int k = 0; k < 8; ++k) z = fmaf(v[k], 0.f, z);
        if (pool) {
          gather(((jj * jstep + 1) * n_col + c) / 4, v2);
#pragma unroll
          for (int k = 0; k < 8; ++k) z = fmaf(v2[k], 0.f, z);
          pool_columns(v, v2);
        }
        const int top = min(n_f, col0 + n_col);
        if (dst >= 0 && z != 0.f && col0 + c < (g.out_p8 ? g.rows - it.f0 : n_f)) redo = 1u;
        finish_columns<HALF, kEither>(g, yv, v, bias_s, dst, it.f0, col0 + c, top, plane, pool, pairs, lane);
      }
      if (HALF && __any_sync(0xffffffffu, redo)) emit_from_lists<HALF, P8>(L, g, 1u, xv, bias, yv, (int)rank, g.parts);
      if (!HALF && redo) redo_s[warp] = 1;
    }
    cluster_sync();      // (nobody leaves while its sums are being read)
  }

  // ---- common exit ----------------------------------------------------------------------------
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (tid == 0) T_STAMP(13);
  if (warp == C::kMmaWarp)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 512;" ::"r"(tmem) : "memory");
  // fp32: where no register is free for it in the roles
  if (!HALF && threadIdx.x < 32 * C::kEpiWarps && redo_s[threadIdx.x >> 5] != 0) {
    uint32_t rank = 0;
    if (g.cluster) asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(rank));
    emit_from_lists<HALF, P8>(L, g, redo_s[threadIdx.x >> 5], xv, bias, yv, (int)rank, g.cluster ? g.parts : 1);
  }
}

// ---- position rows ------------------------------------------------------------------------------
// The activations of a layer as the tensor core reads them: per 8 channels, piece and plane one 16-byte
// row per position of the batch's line (see the top), `lead` zero rows before it and zero rows behind.
struct Rows {
  int pitch, cell_rows, sy, sx;      // positions of a row, rows of an image, row / column parity planes
  int lead, plane_len, groups;       // 8-channel groups: two per 16-channel step
  long long positions;               // of the batch
};

// One thread per (position, group): 8 channel loads, coalesced along the positions, and one 16-byte store
// per piece.  Bound by memory: 4 (2) bytes read and 6 (2) written per fp32 (fp16) value.
template <bool HALF>
__global__ void __launch_bounds__(256) stage_kernel(const Rows r, const void* __restrict__ xv, uint4* __restrict__ out,
                                                    int c_in, int h, int w, int in_sy, int in_sx) {
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  const int at = blockIdx.x * 256 + threadIdx.x;
  constexpr int kPieces = HALF ? 1 : 3;
  const int planes = r.sy * r.sx;
  const int plane = blockIdx.z;
  long long src = -1;
  const int p = at - r.lead;
  if (p >= 0 && p < r.positions) {
    const int R = p / r.pitch, j = p - R * r.pitch;
    const int img = R / r.cell_rows, i = R - img * r.cell_rows;
    const int y = in_sy * i + plane / r.sx, x = in_sx * j + plane % r.sx;
    if (y < h && x < w) src = ((long long)img * c_in * h + y) * w + x;
  }
  asm volatile("griddepcontrol.wait;" ::: "memory");
  if (at >= r.plane_len) return;
  const size_t hw = (size_t)h * w;
  for (int grp = blockIdx.y; grp < r.groups; grp += gridDim.y) {
    const int c0 = grp * 8;
    uint4* o = out + ((size_t)grp * kPieces * planes + plane) * r.plane_len + at;
    const size_t piece = (size_t)planes * r.plane_len;
    uint32_t p1[4], p2[4], p3[4];
    if constexpr (HALF) {
      const unsigned short* s = reinterpret_cast<const unsigned short*>(xv) + (src < 0 ? 0 : src) + (size_t)c0 * hw;
      uint32_t v[8];
#pragma unroll
      for (int i = 0; i < 8; ++i) v[i] = (src >= 0 && c0 + i < c_in) ? (uint32_t)__ldg(s + i * hw) : 0u;
#pragma unroll
      for (int i = 0; i < 4; ++i) p1[i] = v[2 * i] | (v[2 * i + 1] << 16);
      o[0] = make_uint4(p1[0], p1[1], p1[2], p1[3]);
    } else {
      const float* s = reinterpret_cast<const float*>(xv) + (src < 0 ? 0 : src) + (size_t)c0 * hw;
      float v[8];
#pragma unroll
      for (int i = 0; i < 8; ++i) v[i] = (src >= 0 && c0 + i < c_in) ? __ldg(s + i * hw) : 0.f;
#pragma unroll
      for (int i = 0; i < 4; ++i) split_pair(v[2 * i], v[2 * i + 1], p1[i], p2[i], p3[i]);
      o[0] = make_uint4(p1[0], p1[1], p1[2], p1[3]);
      o[piece] = make_uint4(p2[0], p2[1], p2[2], p2[3]);
      o[2 * piece] = make_uint4(p3[0], p3[1], p3[2], p3[3]);
    }
  }
}

Rows rows_of(int c_in, int stride, int n, int h, int w, bool pool) {
  Rows r;
  const int ho = (h - 1) / stride + 1, wo = (w - 1) / stride + 1;
  r.pitch = (wo + 2) / 2 * 2;        // at least one zero column, and even: a lane's neighbour is its row's
  r.cell_rows = (pool ? ho / 2 : ho) + 1;
  r.sy = (stride == 2 || pool) ? 2 : 1;
  r.sx = stride;
  r.lead = r.pitch + 1;
  r.positions = (long long)n * r.cell_rows * r.pitch;
  // an item may end past the batch by up to its 512 positions and the shift of the last tap
  const long long len = r.lead + r.positions + 512 + r.pitch + 2;
  r.plane_len = len > 0x3FFFFFFF ? -1 : (int)len;
  r.groups = 2 * ((c_in + 15) / 16);
  return r;
}
size_t rows_bytes(const Rows& r, bool half) {
  return (size_t)r.groups * (half ? 1 : 3) * r.sy * r.sx * r.plane_len * 16;
}

// ---- launch geometry --------------------------------------------------------------------------

// Cycles of one MMA of 128 x n x 16 (measured: the multiply-adds, or its operands from shared memory).
double mma_cycles(int n) { return n / 2.0 > 32.0 + n / 4.0 ? n / 2.0 : 32.0 + n / 4.0; }

int round_up(int v, int m) { return (v + m - 1) / m * m; }

// Geometry in three steps, each kept while the next is tried with other values: of the map, with `tiles` MMA tiles
// per item, and with nt filters per tile, channel steps not cut.  False where it does not fit.
bool geo_of_map(const DeviceLayer& L, int n, int h, int w, bool pool, bool p8, DGeo* out) {
  DGeo& g = *out;
  g = DGeo{};
  const bool half = L.storage == PCONV_F16;
  const int s = L.stride;
  g.n = n;
  g.h = h;
  g.w = w;
  g.c_in = L.c_in;
  g.c_out = L.c_out;
  const int ho = (h - 1) / s + 1, wo = (w - 1) / s + 1;     // of the convolution itself
  if (pool && s != 1) return false;
  g.pool = pool ? 1 : 0;
  g.h_out = pool ? ho / 2 : ho;
  g.w_out = pool ? wo / 2 : wo;
  // Column strips: a staged slab is an item's positions and a row and a bit on both sides, so a row may
  // not be much longer than an item (128..512 positions).
  g.strips = p8 ? 1 : (wo + 239) / 240;
  g.strip_w = g.strips == 1 ? wo : round_up((wo + g.strips - 1) / g.strips, 2);
  g.strips = (wo + g.strip_w - 1) / g.strip_w;
  g.ox = g.strips > 1 ? 1 : 0;
  g.pitch = round_up(g.strips > 1 ? g.strip_w + 2 : wo + 1, 2);   // even: a lane's neighbour is its row's
  g.cell_rows = g.h_out + 1;
  g.cell_pos = g.cell_rows * g.pitch;
  g.n_cells = n * g.strips;
  fast_div_of(g.cell_pos, &g.cell_mul, &g.cell_shift);
  fast_div_of(g.pitch, &g.pitch_mul, &g.pitch_shift);
  g.sy = (s == 2 || pool) ? 2 : 1;
  g.sx = s;
  g.planes = s == 2 ? 4 : (pool ? 2 : 1);
  if ((long long)g.n_cells * g.cell_pos > 0x3FFFFFFF || (long long)n * L.c_in * h * w > 0x7FFFFFFF) return false;
  // Producers' loads: as many pixels of a row as rows are aligned for (strips start off by one).
  g.vec = 1;
  if (g.strips == 1) g.vec = half && w % 4 == 0 ? 4 : (w % 2 == 0 ? 2 : 1);
  g.row_planes = (s == 2 || pool) ? 2 : 1;
  g.vec_cols = (s * g.pitch + g.vec - 1) / g.vec;
  const Rows in = rows_of(L.c_in, s, n, h, w, pool);
  if (p8 && in.plane_len < 0) return false;
  if (p8) g.vec = 0;
  g.in_plane_len = in.plane_len;
  g.in_lead = in.lead;
  g.rows = L.dense_rows;
  g.n_taps = __builtin_popcount(L.tap_mask);
  g.tps = half ? 3 : 1;
  g.slots = (g.n_taps + g.tps - 1) / g.tps;
  g.k_steps = (L.c_in + 15) / 16;
  return true;
}

bool geo_of_tiles(const DeviceLayer& L, int tiles, DGeo* out) {
  DGeo& g = *out;
  const bool half = L.storage == PCONV_F16, pool = g.pool != 0;
  if ((pool && tiles % 2) || (!half && tiles > 2)) return false;
  g.tiles = tiles;
  g.mpos = pool ? tiles * 64 : tiles * 128;
  // taps: plane and shift
  int plane[kMaxT][9], shift[kMaxT][9], lo = 0, hi = 0, nk = 0;
  for (int t = 0; t < 9; ++t) {
    if (!(L.tap_mask >> t & 1)) continue;
    const int u = t / 3, v = t % 3;
    for (int j = 0; j < tiles; ++j) {
      if (L.stride == 2) {
        plane[j][nk] = (u == 1 ? 0 : 2) + (v == 1 ? 0 : 1);
        shift[j][nk] = (u == 0 ? -g.pitch : 0) + (v == 0 ? -1 : 0) + g.ox;
      } else if (pool) {
        const int r = (j & 1) + u - 1;                 // -1 .. 2
        plane[j][nk] = r & 1;
        shift[j][nk] = (r < 0 ? -1 : r >> 1) * g.pitch + v - 1 + g.ox;
      } else {
        plane[j][nk] = 0;
        shift[j][nk] = (u - 1) * g.pitch + v - 1 + g.ox;
      }
      if (shift[j][nk] < lo) lo = shift[j][nk];
      if (shift[j][nk] > hi) hi = shift[j][nk];
    }
    ++nk;
  }
  g.lead = -lo;
  g.plane_pos = g.mpos + hi - lo;
  g.q_tot = g.planes * g.plane_pos;
  for (int j = 0; j < tiles; ++j)
    for (int t = 0; t < nk; ++t)
      g.tap_off[j][t] = plane[j][t] * g.plane_pos + g.lead + shift[j][t] + 128 * (pool ? j >> 1 : j);
  g.vec_rows = (g.plane_pos + g.pitch - 2) / g.pitch + 1;
  g.n_vec = g.vec ? g.row_planes * g.vec_rows * g.vec_cols : 0;
  g.a_bytes = (half ? 1 : 3) * 2 * g.q_tot * 16;
  g.a_off = round_up(kHeader + kTables * g.n_vec * (int)sizeof(Load), 128);
  return true;
}

bool geo_of_filters(const DeviceLayer& L, int nt, int sms, DGeo* out) {
  DGeo& g = *out;
  const bool half = L.storage == PCONV_F16, p8 = g.vec == 0;
  const int tiles = g.tiles;
  g.nt = nt;
  g.n_ft = (g.rows + nt - 1) / nt;
  g.form3 = (!half && 3 * nt <= 256 && tiles * 3 * nt <= 512) ? 1 : 0;
  g.tile_cols = half ? nt : (g.form3 ? 3 : 2) * nt;
  g.n_buf = (half && tiles * nt <= 256) ? 2 : 1;
  if (tiles * g.tile_cols > 512 || nt > 128 || (!half && tiles * nt > (p8 ? 256 : 128))) return false;
  g.out_col = !half && tiles * (g.tile_cols + nt) <= 512 ? tiles * g.tile_cols : 0;
  g.out_stride = g.out_col ? nt : g.tile_cols;
  // the epilogue reads columns by 16, which may pass the end of a tile but not Tensor Memory's
  if (half && (g.n_buf == 2 ? 256 : 0) + (tiles - 1) * nt + nt / 2 + round_up(nt / 2, 16) > 512) return false;
  if (!half && (tiles - 1) * g.tile_cols + (g.form3 ? 2 : 1) * nt + nt / 2 + round_up(nt / 2, 16) > 512) return false;
  g.b_bytes = g.tps * (half ? 1 : 3) * 2 * nt * 16;
  const int avail = kSmemLimit - g.a_off;
  // Activation stages first (two, so that one is filled while the other is read), then as many weight
  // slots as fit: what matters there is the time of the MMAs they cover against a copy's latency.
  g.a_stages = 2;
  if (2 * g.a_bytes + 8 * g.b_bytes > avail) g.a_stages = 1;
  while (g.a_stages < kMaxA && (g.a_stages + 1) * g.a_bytes + (half ? 8 : 16) * g.b_bytes <= avail) ++g.a_stages;
  g.b_slots = (avail - g.a_stages * g.a_bytes) / g.b_bytes;
  if (g.b_slots > kMaxB) g.b_slots = kMaxB;
  if (g.b_slots < (half ? 3 : 7)) return false;
  g.b_off = g.a_off + g.a_stages * g.a_bytes;
  const long long m_items = ((long long)g.n_cells * g.cell_pos + g.mpos - 1) / g.mpos;
  const long long items = m_items * g.n_ft;
  if (items > 0x3FFFFF || items * g.k_steps > 0x3FFFFFFF) return false;
  g.n_tiles = (int)items;
  g.grid = std::min(g.n_tiles, sms);
  return true;
}

// Workspace of a split launch: fp32 sums of the tiles that may be cut, then their tickets.
size_t slots(const DGeo& g) { return std::min(g.grid, g.n_tiles); }
size_t sums_bytes(const DGeo& g) { return slots(g) * g.tiles * g.nt * 128 * sizeof(float); }
size_t split_bytes(const DGeo& g) {
  return g.split && !g.cluster ? sums_bytes(g) + ((slots(g) * 8 * sizeof(int) + 255) & ~(size_t)255) : 0;
}

// Estimated cycles of a launch.  A step lasts as long as its MMAs, its share of the weight stream (about
// 36 bytes a cycle and SM from L2) or the staging of its activations, whichever is longest; an item ends with
// its stores, which only the fp32 kernel and two accumulator sets overlap with the next item; a split adds
// the exchange of partial sums.
struct StepCost {
  double step, epi;      // a channel step of an item, and its end
};
double tap_cycles(const DGeo& g, bool half) {      // the MMAs of a tap of one tile
  const int nt = g.nt;
  return half ? mma_cycles(nt)
              : (g.form3 ? mma_cycles(3 * nt) + mma_cycles(2 * nt) + mma_cycles(nt) : mma_cycles(2 * nt) + 4 * mma_cycles(nt));
}
StepCost step_cost(const DGeo& g, bool half) {
  const int nt = g.nt;
  double step = tap_cycles(g, half) * g.n_taps * g.tiles;
  const double wb = ((double)g.n_taps * (half ? 1 : 3) * nt * 32 + (g.vec ? 0.0 : g.a_bytes)) / 36.0;
  // (a batch of the producers -- a load and its rows a thread -- takes about as long whatever its width)
  double conv = 300.0 + (half ? 1100.0 : 1300.0) * ((2 * g.n_vec + 319) / 320);
  if (!g.vec) conv = 60.0 * (half ? 2 : 6) * g.planes;      // one bulk copy each
  if (wb > step) step = wb;
  if (conv > step) step = conv;
  step += 60;
  return {step, 600 + (half ? 8.0 : 16.0) * g.tiles * nt};
}
long long ceil_div(long long a, long long b) { return (a + b - 1) / b; }
long long steps_of(const DGeo& g) {                // channel steps of the CTA that has most of them
  return g.split ? ceil_div((long long)g.n_tiles * g.k_steps, g.grid) : ceil_div(g.n_tiles, g.grid) * g.k_steps;
}
double dense_cycles(const DGeo& g, const StepCost& cost, bool half, int sms) {
  const int nt = g.nt;
  const double epi = cost.epi;
  const long long steps = steps_of(g);
  const long long segments = ceil_div(steps, g.k_steps);
  double c = 4500 + steps * cost.step + epi + (segments - 1) * (half && g.n_buf == 1 ? epi : 0.25 * epi);
  if (g.split) {
    // A part hands its sums over, inside a cluster or added to the workspace.  Measured on layers of 49 to
    // 3136 positions: a cluster's exchange 5000-6000 cycles, more where large clusters have to wait for
    // neighbouring SMs; the workspace's about as much up to some 30 KB per SM, then reductions of all SMs
    // together run at about 1 TB/s.  An uneven split goes through it twice.
    const double bytes = (double)g.tiles * nt * 512;
    if (g.cluster) c += 4700 + bytes / 24.0 + (g.parts > 4 ? 800.0 : 0.0) + (g.parts >= 4 && 2 * g.grid > sms ? 1500.0 : 0.0);
    else c += (4200 + bytes * g.grid / sms / 8.0) * (g.parts ? 1.0 : 2.0);
  }
  return c;
}
// What a launch is expected to take, in microseconds.  dense_cycles ranks the plans of one shape; this sets a plan
// against the sparse kernel, for which a rank is not enough.  Constants fitted (least squares of log ratios, both
// strides, 3 to 512 channels, 16 to 512 filters, maps of 4 to 112 pixels, 1 to 64 images) to 4826 layers timed
// in every form: measured over expected has a standard deviation of 0.07 for fp32 and 0.09 for fp16, where
// dense_cycles has 0.19 and 0.21.  What it has that dense_cycles has not: with a single activation stage a
// step's copies or conversions come after its MMAs.
double launch_us(const DGeo& g, bool half) {
  struct Fit {   // cycles of 0.6 ns; rates in bytes a cycle
    double base_nchw, base_rows, step, mma, copy_rate, conv0, conv1, epi0, epi1, more, exchange, part, cluster_rate, ws_rate;
  };
  static const Fit kFit[2] = {
      {787, 2335, 1699, 0.619, 81.0, 69, 733, 7824, 67.9, 0.416, 2860, 13.4, 18.7, 7.15},
      {5113, 4256, 771, 0.467, 74.5, 0, 734, 906, 40.8, 0.655, 2919, 0.0, 15.3, 9.45}};
  const Fit& f = kFit[half ? 1 : 0];
  const bool p8 = g.vec == 0;
  const double copies = (double)g.n_taps * (half ? 1 : 3) * g.nt * 32 + (p8 ? g.a_bytes : 0);
  const double fill = p8 ? g.a_bytes / f.copy_rate : f.conv0 + f.conv1 * ((2 * g.n_vec + 319) / 320);
  double step = std::max(tap_cycles(g, half) * g.n_taps * g.tiles * f.mma, copies / f.copy_rate);
  step = (g.a_stages == 1 ? step + fill : std::max(step, fill)) + f.step;
  const long long steps = steps_of(g), segments = ceil_div(steps, g.k_steps);
  double c = (p8 ? f.base_rows : f.base_nchw) + steps * step + (f.epi0 + f.epi1 * g.tiles * g.nt) * (1 + (segments - 1) * f.more);
  const double bytes = (double)g.tiles * g.nt * 512;
  if (g.cluster) c += f.exchange + f.part * g.parts + bytes / f.cluster_rate;
  else if (g.split) c += (f.exchange + bytes * g.grid / 148 / f.ws_rate) * (g.parts ? 1 : 2);
  return 6e-4 * c;
}
// What no way of cutting these tiles can fall below: all steps spread evenly over all SMs.
double least_cycles(const DGeo& g, const StepCost& cost, int sms) {
  return 4500 + ceil_div((long long)g.n_tiles * g.k_steps, sms) * cost.step + cost.epi;
}

int max_clusters(int dev, bool half, int parts);   // below: needs the kernels
#ifdef PCONV_DEV
std::atomic<long long> g_plans_made{0};
#endif

// The geometry of a launch: the cheapest by the estimate.  ws_bytes: workspace the caller has; sms, clusters(parts):
// the device's.  `prune`: what cannot become the cheapest is left out before its ways of cutting are gone through,
// which changes no plan.
template <typename Clusters>
bool dense_plan(const DeviceLayer& L, int n, int h, int w, bool pool, bool p8, size_t ws_bytes, int sms, Clusters clusters,
                bool prune, DGeo* out, double* cycles) {
  const bool half = L.storage == PCONV_F16;
  bool found = false;
  double best = 0.0;
#ifdef PCONV_DEV
  ++g_plans_made;
  int force[4] = {0, 0, 0, 0};
  if (const char* e = getenv("PCONV_FORCE_DENSE")) sscanf(e, "%d,%d,%d,%d", &force[0], &force[1], &force[2], &force[3]);
#endif
  DGeo of_tiles[3];                              // 1, 2 and 4 tiles
  bool fits[3];
  if (!geo_of_map(L, n, h, w, pool, p8, &of_tiles[0])) return false;
  of_tiles[1] = of_tiles[2] = of_tiles[0];
  for (int t = 0; t < 3; ++t) fits[t] = geo_of_tiles(L, 1 << t, &of_tiles[t]);
  int last_nt = 0;
  for (int cut = (L.dense_rows + 127) / 128; cut <= L.dense_rows / 16; cut = cut < 4 ? cut + 1 : cut * 2) {
    const int nt = round_up((L.dense_rows + cut - 1) / cut, 16);
    if (nt == last_nt || nt > 128) continue;
    last_nt = nt;
    if (nt < 32 && L.dense_rows > 16) break;
    for (int t = 0; t < 3; ++t) {
      DGeo g = of_tiles[t];
      if (!fits[t] || !geo_of_filters(L, nt, sms, &g)) continue;
      const StepCost cost = step_cost(g, half);
      if (prune && found && least_cycles(g, cost, sms) >= best) continue;
      // Whole tiles only (v = 0); or the line of steps cut evenly among all SMs (1); or each tile cut in
      // v / 2 parts, a CTA's each: in the workspace (even v; equal parts, which end together) or, up to
      // eight, by a cluster, which needs none.
      const int whole = g.grid;
      for (int v = 0; v <= 2 * (g.k_steps / kMinSteps) + 1; ++v) {
        const int parts = v < 2 ? v : v / 2;
        g.grid = whole;
        g.split = g.cluster = 0;
        if (parts == 1) {
          if (v != 1 || g.n_tiles % sms == 0 || g.k_steps < 2 * kMinSteps) continue;
          g.grid = (int)std::min<long long>(sms, (long long)g.n_tiles * (g.k_steps / kMinSteps));
          g.split = 1;
        } else if (parts > 1) {
          if ((long long)g.n_tiles * parts > sms || g.k_steps < kMinSteps * parts) break;
          g.grid = g.n_tiles * parts;
          g.split = 1;
          g.cluster = v & 1;
          if (!g.cluster && g.k_steps % parts != 0) continue;
          if (g.cluster && (parts > 8 || g.n_tiles > clusters(parts) ||
                            g.tiles * nt * 512 > g.a_stages * g.a_bytes + g.b_slots * g.b_bytes))
            continue;
        }
        if (split_bytes(g) > ws_bytes) continue;
        const int all = g.split ? g.n_tiles * g.k_steps : g.n_tiles;
        g.share = all / g.grid;
        g.share_more = all % g.grid;
        g.parts = g.cluster ? parts : g.split && g.share_more == 0 && g.k_steps % g.share == 0 ? g.k_steps / g.share : 0;
        double c = dense_cycles(g, cost, half, sms);
#ifdef PCONV_DEV
        if (force[0] && (force[0] != g.tiles || force[1] != nt || force[2] != g.grid || force[3] != g.cluster)) c += 1e12;
#endif
        if (!found || c < best) {
          found = true;
          best = c;
          *out = g;
        }
      }
    }
  }
  if (found) *cycles = best;
  return found;
}

// The plans of recent launches, one table for the process: planning takes microseconds, a repeated call finds its
// plan in a tenth of one.  A plan is kept by all that it depends on, which is a layer's geometry and not the
// layer (ResNet-50's sixteen 3x3 layers have seven), and for every workspace from the one it needs up to
// the one it was made for: what was the cheapest of more choices is the cheapest of fewer.
struct PlanKey {
  int c_in, c_out, stride, storage, tap_mask, n, h, w, form, dev;      // form: 2 pool + position rows
};
struct Plan {
  bool found;
  double cycles, us;           // rank and expected time
  size_t need;                 // workspace
  int n_tiles, n_ft;
};
struct PlanEntry {
  PlanKey key;
  size_t most;                 // it holds for workspaces from plan.need to this
  Plan plan;
  DGeo geo;
};
constexpr int kPlanSets = 64, kPlanWays = 8;       // (the oldest of a set is replaced)
struct PlanTable {
  std::mutex lock;
  PlanEntry entry[kPlanSets][kPlanWays];           // (zeroed: no key has n = 0)
  unsigned char next[kPlanSets];
};
PlanTable g_plans;

PlanKey plan_key(const DeviceLayer& L, int n, int h, int w, bool pool, bool p8) {
  int dev = -1;
  if (cudaGetDevice(&dev) != cudaSuccess) cudaGetLastError();
  return {L.c_in, L.c_out, L.stride, L.storage, L.tap_mask, n, h, w, 2 * (int)pool + (int)p8, dev};
}
int plan_set(const PlanKey& k, unsigned long long hash) {
  for (int v : {k.c_in, k.c_out, k.n, k.h, k.w, (k.tap_mask << 8) + (k.form << 4) + (k.stride << 2) + k.storage})
    hash = (hash ^ (unsigned)v) * 0x9E3779B97F4A7C15ull, hash ^= hash >> 29;
  return (int)((hash >> 40) % kPlanSets);
}

Plan find_plan(const DeviceLayer& L, int n, int h, int w, bool pool, bool p8, size_t ws_bytes, DGeo* geo = nullptr) {
  if (!L.wdense || n <= 0 || h <= 0 || w <= 0) return Plan{};
  if (ws_bytes > kMaxSplitBytes) ws_bytes = kMaxSplitBytes;
  const PlanKey k = plan_key(L, n, h, w, pool, p8);
  const int set = plan_set(k, 0);
#ifdef PCONV_DEV
  const bool keep = !getenv("PCONV_FORCE_DENSE");      // (a forced plan is nobody else's)
#else
  const bool keep = true;
#endif
  if (keep) {
    std::lock_guard<std::mutex> hold(g_plans.lock);
    for (const PlanEntry& e : g_plans.entry[set])
      if (std::memcmp(&e.key, &k, sizeof(k)) == 0 && ws_bytes >= e.plan.need && ws_bytes <= e.most) {
        if (geo) *geo = e.geo;
        return e.plan;
      }
  }
  PlanEntry made = {};
  DGeo& g = made.geo;
  made.key = k;
  made.most = ws_bytes;
  const bool half = L.storage == PCONV_F16;
  made.plan.found = dense_plan(L, n, h, w, pool, p8, ws_bytes, device_sm_count(),
                               [&](int parts) { return max_clusters(k.dev, half, parts); }, true, &g, &made.plan.cycles);
  if (made.plan.found) {
    made.plan.need = split_bytes(g);
    made.plan.us = launch_us(g, half);
  }
  made.plan.n_tiles = g.n_tiles;
  made.plan.n_ft = g.n_ft;
#ifdef PCONV_DEV
  if (made.plan.found && getenv("PCONV_DENSE_VERBOSE"))
    fprintf(stderr, "dense %d->%d %dx%d n%d s%d pool%d p8 %d ws%zu: tiles %d nt %d split %d cluster %d grid %d n_tiles %d q %d pitch %d a_stages %d b_slots %d cycles %.0f us %.1f\n",
            L.c_in, L.c_out, h, w, n, L.stride, (int)pool, (int)p8, ws_bytes, g.tiles, g.nt, g.split, g.cluster * g.parts, g.grid,
            g.n_tiles, g.q_tot, g.pitch, g.a_stages, g.b_slots, made.plan.cycles, made.plan.us);
#endif
  if (geo) *geo = g;
  if (keep) {
    std::lock_guard<std::mutex> hold(g_plans.lock);
    g_plans.entry[set][g_plans.next[set]++ % kPlanWays] = made;
  }
  return made.plan;
}

// Zero-inserted weights from the per-filter lists: one block per filter, one thread per kernel.  Layout:
// [channel step of 16][stored tap][8 channels][piece][filter row][8] (bf16 pieces, or the fp16 values).
__global__ void __launch_bounds__(128) dense_weights_kernel(const DeviceLayer L) {
  const int o = blockIdx.x;
  const bool half = L.storage == PCONV_F16;
  const int pieces = half ? 1 : 3;
  const int n_taps = __popc(L.tap_mask);
  unsigned short* wd = reinterpret_cast<unsigned short*>(const_cast<void*>(L.wdense));
  for (int k = L.row_ptr[o] + threadIdx.x; k < L.row_ptr[o + 1]; k += blockDim.x) {
    const uint32_t idx = L.csr_idx[k];
    const int c = idx & 0xFFFF;
    const uint32_t mask = idx >> 16;
    int s = 0;
    for (int t = 0; t < 9; ++t) {
      if (!(mask >> t & 1)) continue;
      const float v = L.csr_val[4 * k + s++];
      const int ti = __popc(L.tap_mask & ((1 << t) - 1));
      const size_t run = ((size_t)(c / 16) * n_taps + ti) * (2 * pieces) + (size_t)((c >> 3) & 1) * pieces;
      unsigned short* d = wd + (run * L.dense_rows + o) * 8 + (c & 7);
      if (half) {
        *d = __half_as_ushort(__float2half_rn(v));
      } else {
        float rest = v;
        for (int p = 0; p < 3; ++p) {
          uint32_t piece = (__float_as_uint(rest) + 0x8000u) & 0xFFFF0000u;
          if ((piece & 0x7F800000u) == 0x7F800000u) piece -= 0x10000u;    // (packed weights are finite)
          d[(size_t)p * L.dense_rows * 8] = (unsigned short)(piece >> 16);
          rest -= __uint_as_float(piece);
        }
      }
    }
  }
}

// Clusters of `parts` CTAs that the device holds at once (one CTA per SM, the SMs of a cluster inside one
// GPC); asked once per size and device (`dev`: the current one).  Without a device: none.
int max_clusters(int dev, bool half, int parts) {
  static std::atomic<int> known[64][2][9];
  if (dev < 0 || dev >= 64) return 0;
  std::atomic<int>& slot = known[dev][half ? 1 : 0][parts];
  int v = slot.load();
  if (v) return v - 1;
  const void* f = half ? (const void*)dense_kernel<true, 0> : (const void*)dense_kernel<false, 0>;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)parts, 1, 1);
  cfg.blockDim = dim3(Cfg<false, true>::kThreads, 1, 1);
  cfg.dynamicSmemBytes = kSmemLimit;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = (unsigned)parts;
  attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  int n = 0;
  if (cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemLimit) != cudaSuccess ||
      cudaOccupancyMaxActiveClusters(&n, f, &cfg) != cudaSuccess) {
    cudaGetLastError();
    n = 0;
  }
#ifdef PCONV_DEV
  if (getenv("PCONV_DENSE_VERBOSE")) fprintf(stderr, "clusters of %d: %d\n", parts, n);
#endif
  slot.store(n + 1);
  return n;
}

template <bool HALF, int V>
cudaError_t launch_dense_geo(const DeviceLayer& L, const DGeo& g, const void* x, const float* bias, void* y, float* ws,
                             int* tickets, cudaStream_t stream) {
  static std::atomic<bool> ready[64];
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev >= 64 || !ready[dev]) {
    e = cudaFuncSetAttribute(dense_kernel<HALF, V>, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemLimit);
    if (e != cudaSuccess) return e;
    if (dev < 64) ready[dev] = true;
  }
  const int smem = g.b_off + g.b_slots * g.b_bytes;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)g.grid, 1, 1);
  cfg.blockDim = dim3(Cfg<HALF, V == 0>::kThreads, 1, 1);
  // more than half of an SM's shared memory: one CTA per SM (each takes all of Tensor Memory)
  cfg.dynamicSmemBytes = (size_t)(smem < 120 * 1024 ? 120 * 1024 : smem);
  cfg.stream = stream;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  attr[1].id = cudaLaunchAttributeClusterDimension;
  attr[1].val.clusterDim.x = (unsigned)g.parts;
  attr[1].val.clusterDim.y = attr[1].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = g.cluster ? 2 : 1;
  return cudaLaunchKernelEx(&cfg, dense_kernel<HALF, V>, L, g, x, bias, y, ws, tickets);
}

}  // namespace

size_t dense_weight_bytes(const DeviceLayer& L) {
  const size_t pieces = L.storage == PCONV_F16 ? 1 : 3;
  return (size_t)((L.c_in + 15) / 16) * __builtin_popcount(L.tap_mask) * 2 * pieces * L.dense_rows * 16;
}

cudaError_t dense_build_weights(const DeviceLayer& L, cudaStream_t stream) {
  cudaError_t e = cudaMemsetAsync(const_cast<void*>(L.wdense), 0, dense_weight_bytes(L), stream);
  if (e != cudaSuccess) return e;
  dense_weights_kernel<<<L.c_out, 128, 0, stream>>>(L);
  return cudaGetLastError();
}

// (whether there is a plan does not depend on the workspace: whole tiles need none)
bool dense_supported(const DeviceLayer& L, int n, int h, int w, bool pool, size_t ws_bytes) {
  return find_plan(L, n, h, w, pool, false, ws_bytes).found;
}

size_t dense_workspace_bytes(const DeviceLayer& L, int n, int h, int w, bool pool, RowsFrom rows, size_t most) {
  size_t need = find_plan(L, n, h, w, pool, false, most).need;
  if (rows == kRowsGiven || dense_path(L, n, h, w, pool, rows, most) == kFromRows)
    need = std::max(need, find_plan(L, n, h, w, pool, true, most).need);
  return need;
}

bool dense_takes_rows(const DeviceLayer& L, int n, int h, int w, bool pool, size_t ws_bytes) {
  return find_plan(L, n, h, w, pool, true, ws_bytes).found;
}

size_t dense_rows_bytes(const DeviceLayer& L, int n, int h, int w, bool pool) {
  return rows_bytes(rows_of(L.c_in, L.stride, n, h, w, pool), L.storage == PCONV_F16);
}

size_t dense_scratch_bytes(const DeviceLayer& L, int n, int h, int w, bool pool, size_t ws_bytes) {
  // (dense_path_alone takes a choice back, but makes none: it need not be asked where rows are not chosen)
  return dense_path(L, n, h, w, pool, kRowsStaged, ws_bytes) == kFromRows &&
                 dense_path_alone(L, n, h, w, pool, kRowsStaged, ws_bytes) == kFromRows
             ? dense_rows_bytes(L, n, h, w, pool) : 0;
}

cudaError_t launch_stage(const DeviceLayer& L, const void* x, void* rows, int n, int h, int w, bool pool,
                         cudaStream_t stream) {
  const Rows r = rows_of(L.c_in, L.stride, n, h, w, pool);
  cudaLaunchConfig_t cfg = {};
  const int blocks = (r.plane_len + 255) / 256, planes = r.sy * r.sx;
  // groups share the position arithmetic of a thread once the device is full without them
  int gy = r.groups;
  while (gy > 1 && (long long)blocks * planes * gy > 32ll * device_sm_count()) gy = (gy + 1) / 2;
  cfg.gridDim = dim3((unsigned)blocks, (unsigned)gy, (unsigned)planes);
  cfg.blockDim = dim3(256, 1, 1);
  cfg.stream = stream;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return L.storage == PCONV_F16
             ? cudaLaunchKernelEx(&cfg, stage_kernel<true>, r, x, (uint4*)rows, L.c_in, h, w, r.sy, r.sx)
             : cudaLaunchKernelEx(&cfg, stage_kernel<false>, r, x, (uint4*)rows, L.c_in, h, w, r.sy, r.sx);
}

cudaError_t launch_dense(const DeviceLayer& L, const void* x, const float* bias, void* y, int n, int h, int w,
                         bool relu, bool pool, bool rows_in, const DenseNext* next, void* ws, size_t ws_bytes,
                         cudaStream_t stream) {
  DGeo g;
  if (!find_plan(L, n, h, w, pool, rows_in, ws ? ws_bytes : 0, &g).found) return cudaErrorInvalidValue;
  g.relu = relu ? 1 : 0;
  if (next) {
    const Rows r = rows_of(next->c_in, next->stride, n, g.h_out, g.w_out, next->pool);
    g.out_p8 = 1;
    g.out_pitch = r.pitch;
    g.out_cell_rows = r.cell_rows;
    g.out_sy = r.sy;
    g.out_sx = r.sx;
    g.out_plane_len = r.plane_len;
    g.out_lead = r.lead;
  }
  float* sums = g.split ? (float*)ws : nullptr;
  int* tickets = g.split ? (int*)((char*)ws + sums_bytes(g)) : nullptr;
  if (L.storage == PCONV_F16) {
    if (rows_in) return launch_dense_geo<true, 0>(L, g, x, bias, y, sums, tickets, stream);
    if (g.vec == 4) return launch_dense_geo<true, 4>(L, g, x, bias, y, sums, tickets, stream);
    if (g.vec == 2) return launch_dense_geo<true, 2>(L, g, x, bias, y, sums, tickets, stream);
    return launch_dense_geo<true, 1>(L, g, x, bias, y, sums, tickets, stream);
  }
  if (rows_in) return launch_dense_geo<false, 0>(L, g, x, bias, y, sums, tickets, stream);
  if (g.vec == 2) return launch_dense_geo<false, 2>(L, g, x, bias, y, sums, tickets, stream);
  return launch_dense_geo<false, 1>(L, g, x, bias, y, sums, tickets, stream);
}

// What is expected to run this shape fastest: both kernels by estimate.  Sparse kernel: a fixed 12 us, 8 ns a
// channel, twice that at stride 2 (measured at 1 image: 14-15 us at 64-128 channels, 18-23 us at 512) and a
// fifth of the FP32 peak (15-29 % of it in large launches).  Dense kernel: its plan's cycles at 1380 a microsecond,
// which is coarse: 1113 fp32 chains of equal layers took 0.97-1.76 of that (5th to 95th percentile, median
// 1.32; 1.5 at 32 filters a tile, 1.0 at 128), the stress layers of 64 images 1.08 (stride 1) and 1.22.  Staging the input as position rows is a launch of its own and moves every value twice.  Where a
// tile's positions are all there are, each dense weight (54 bytes for fp32, a kept kernel's sparse ones take 6
// a weight) is read for one use and, in a network of such layers, from memory: 512->512 7x7 takes 15 us alone
// and 20-26 us among its neighbours, the sparse kernel 18 us in both.
DensePath dense_path(const DeviceLayer& L, int n, int h, int w, bool pool, RowsFrom rows, size_t ws_bytes) {
  const bool half = L.storage == PCONV_F16;
  const double macs = 4.0 * (double)L.n_kept * n * ((h - 1) / L.stride + 1) * ((w - 1) / L.stride + 1);
  double best = 1380.0 * (12.0 + 0.008 * L.c_in * L.stride + 2.0 * macs / (0.2 * 74.45e6));
  DensePath path = kNotDense;
  auto cycles_of = [&](const Plan& e) {
    return e.cycles + (e.n_tiles <= e.n_ft ? (double)dense_weight_bytes(L) / 1600.0 : 0.0);
  };
#ifdef PCONV_DEV
  if (getenv("PCONV_FORCE_DENSE")) best = 1e15;
  if (const char* f = getenv("PCONV_FORCE_ROWS")) rows = atoi(f) && rows != kNoRows ? kRowsGiven : kNoRows;
#endif
  if (rows != kRowsGiven) {
    const Plan e = find_plan(L, n, h, w, pool, false, ws_bytes);
    if (e.found && cycles_of(e) < best) {
      best = cycles_of(e);
      path = kFromNchw;
    }
  }
  const double staging = rows != kRowsStaged ? 0.0 :
      5500.0 + ((double)rows_bytes(rows_of(L.c_in, L.stride, n, h, w, pool), half) +
                (double)n * L.c_in * h * w * (half ? 2 : 4)) / 2200.0;
  // (no plan where staging the input alone leaves too little: no launch is estimated below 5100 cycles)
  if (rows != kNoRows && staging + 5100.0 < best) {
    const Plan e = find_plan(L, n, h, w, pool, true, ws_bytes);
    if (e.found && cycles_of(e) + staging < best) path = kFromRows;
  }
  return path;
}

double path_us(const DeviceLayer& L, int n, int h, int w, bool pool, DensePath path, bool staged, size_t ws_bytes) {
  if (path == kNotDense) return tiled_us(L, n, h, w, ws_bytes);
  const Plan e = find_plan(L, n, h, w, pool, path == kFromRows, ws_bytes);
  // (laying the input out overlaps its neighbours and moves 6.5 TB/s)
  const double moved = (double)rows_bytes(rows_of(L.c_in, L.stride, n, h, w, pool), L.storage == PCONV_F16);
  return e.us + (path == kFromRows && staged ? 1.0 + moved / 6.5e6 : 0.0);
}

namespace {
// The choices of recent calls, kept as the plans are.
struct ChoiceKey {
  PlanKey shape;
  int rows, codes;
  long long kept;
  size_t ws_bytes;
};
struct ChoiceTable {
  std::mutex lock;
  struct Entry {
    ChoiceKey key;
    DensePath path;
  } entry[kPlanSets][kPlanWays];
  unsigned char next[kPlanSets];
};
ChoiceTable g_choices;

}  // namespace

// dense_path's estimates are coarse (a fifth either way) and favour the dense kernel, which pays in a stack, where each
// dense layer hands the next its input.  A layer of its own that they give to the dense kernel goes back where the
// two expected times (path_us) say that the sparse kernel is faster by more than they are off.  Of 3653 fp32 layers
// 4.9 % instead of 8.2 % then run over 3 % slower than on the sparse kernel, and 0.3 % over 3 % slower than before
// (256->256 28x28 N=2: dense 32.6 us, sparse 24.0).  (The expected times alone, without a margin: 3 % faster over all
// layers timed one by one, but ResNet-50 N=32, whose layers follow one another, 855 -> 887 us.)
DensePath dense_path_alone(const DeviceLayer& L, int n, int h, int w, bool pool, RowsFrom rows, size_t ws_bytes) {
  if (!L.wdense || n <= 0 || h <= 0 || w <= 0) return kNotDense;
#ifdef PCONV_DEV
  if (getenv("PCONV_FORCE_DENSE") || getenv("PCONV_FORCE_ROWS")) return dense_path(L, n, h, w, pool, rows, ws_bytes);
#endif
  ChoiceKey k;
  std::memset(&k, 0, sizeof(k));
  k.shape = plan_key(L, n, h, w, pool, false);
  k.rows = rows;
  k.codes = (L.codes_s ? 2 : 0) + (L.wide_codes ? 1 : 0);
  k.kept = L.n_kept;
  k.ws_bytes = std::min(ws_bytes, kMaxSplitBytes);
  const int set = plan_set(k.shape, (unsigned long long)k.kept * 8 + (unsigned)rows);
  {
    std::lock_guard<std::mutex> hold(g_choices.lock);
    for (const ChoiceTable::Entry& e : g_choices.entry[set])
      if (std::memcmp(&e.key, &k, sizeof(k)) == 0) return e.path;
  }
  DensePath path = dense_path(L, n, h, w, pool, rows, ws_bytes);
  if (path != kNotDense) {
    const double sparse_us = path_us(L, n, h, w, pool, kNotDense, false, ws_bytes);
    if (sparse_us > 0.0 && path_us(L, n, h, w, pool, path, rows == kRowsStaged, ws_bytes) > 1.15 * sparse_us) path = kNotDense;
  }
  std::lock_guard<std::mutex> hold(g_choices.lock);
  ChoiceTable::Entry& e = g_choices.entry[set][g_choices.next[set]++ % kPlanWays];
  e.key = k;
  e.path = path;
  return path;
}

#ifdef PCONV_DEV
bool dense_plan_of_shape(const DeviceLayer& L, int n, int h, int w, bool pool, bool p8, size_t ws_bytes, int cluster_sms,
                         bool prune, int* out, double* cycles) {
  DGeo g = {};
  if (!dense_plan(L, n, h, w, pool, p8, ws_bytes, 148, [&](int parts) { return cluster_sms / parts; }, prune, &g, cycles))
    return false;
  const int f[14] = {g.tiles, g.nt, g.grid, g.split, g.cluster, g.parts, g.n_tiles, g.k_steps, g.a_stages, g.b_slots,
                     g.b_off + g.b_slots * g.b_bytes, g.tiles * g.tile_cols, (int)split_bytes(g), g.share};
  for (int i = 0; i < 14; ++i) out[i] = f[i];
  return true;
}
long long dense_plans_made() { return g_plans_made.load(); }

cudaError_t dense_set_withhold(int step, unsigned spin_limit) {
  const unsigned limit = step >= 0 ? spin_limit : kSpinLimit;
  cudaError_t e = cudaMemcpyToSymbol(g_withhold_step, &step, sizeof(step));
  if (e == cudaSuccess) e = cudaMemcpyToSymbol(g_spin_limit, &limit, sizeof(limit));
  return e;
}
#endif

}  // namespace pconv
