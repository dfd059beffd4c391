// Chunkwise-parallel prefill on the 5th-generation tensor cores (bf16 io, d = 128).
//
// Sec. 4.1: the sequence is cut into non-overlapping groups; inside a group the causally
// masked product phi(Q) phi(K)^T V is formed in parallel, between groups only the cumulative
// sums S = sum phi(k) v^T and z = sum phi(k) are carried.  One CTA walks one (batch, head)
// chain in tiles of 128 tokens:
//     O = phi(Q) S_prev + (P o M) V,   den = phi(Q) . z_prev + rowsum(P o M),   S += phi(K)^T V,   z += colsum phi(K).
// The matrix products run on the tensor cores, and z rides along with them: V is extended by a column of ones
// ([S | z] += phi(K)^T [V | 1], one product of 144 columns), and the K tile by a row that holds z_prev, so
// that the score product delivers phi(q) . z_prev as one more column of P.  The row sums of the masked P are taken
// by the threads that mask it.  Per tile n:
//
//   TMA      Q, K, V tiles (128 x 128 bf16, two 64-column boxes each, 128-byte swizzle)
//   group A  phi(Q) -> TMEM and phi(K) in place (packed bf16x2 arithmetic)
//   tcgen05  [P | phi(q) . z_prev] = phi(Q) [phi(K); z_prev]^T     (144 columns: 128 tokens, z_prev, 15 unused)
//            [S | z] += phi(K)^T [V | 1]               (fp32 in TMEM for the whole chain)
//            O = phi(Q) S_prev                         (S_prev is a bf16 copy in shared memory)
//   group A  phi on K of tile n+1 (K is double-buffered), while the tensor cores form the scores;
//            P -> causal mask, row sums (+ the z column), bf16 -> TMEM (the A operand of the next product)
//   group B  S -> bf16 copy, z -> the K buffer of tile n+1 (long windows: group A)
//   tcgen05  O += (P o M) V
//   group B  o = O / (den + eps) + conv(V) -> the tile's V buffer;  TMA stores it to global memory
// (More than 5 taps: a second epilogue, which forms the tap sums by channel pair and stages the outputs in the tile's
// K buffer; three-branch mode, GRP: the score product on the raw q and k and a causal softmax instead of the mask.)
//
// Five roles run concurrently: group A (warps 8-15), group B (warps 0-7), warp 16, whose elected lane issues
// every MMA and the Q loads, warp 17, one lane of which issues the V loads and the output stores (a store has
// to have read its buffer before the buffer is reloaded: that wait must not hold up the products) and another the
// K reloads, and warp 18, which copies aside the rows of v that the convolution reaches back to.  While group B finishes
// tile n, group A already works on tile n+1.  Every wait on an mbarrier is bounded; when one runs out the CTA
// records LA_ERR_TIMEOUT, stops issuing work, frees its TMEM and returns.
#include <cuda.h>

#include <algorithm>
#include <type_traits>

#include "la_common.cuh"

namespace la {
namespace tc {

constexpr int D = 128;
constexpr int TILE = 128;
constexpr int kThreadsB = 256;                     // group B: warps 0-7
constexpr int kThreadsA = 256;                     // group A: warps 8-15
constexpr int kCtrlWarp = 16, kCopyWarp = 17, kHaloWarp = 18;
constexpr int kThreads = 640;
constexpr uint32_t BOX_BYTES = 128 * 128;          // 128 rows x 64 bf16
constexpr uint32_t TILE_BYTES = 2 * BOX_BYTES;
// A K buffer carries 8 more rows below the 128 token rows of each box, the first of which (row 128) holds z_prev as
// bf16: the score product runs with N = 144 and its column 128 is phi(q) . z_prev.  Columns 129-143 are never read,
// so rows 129-135 hold whatever they hold and rows 136-143 are simply the first kilobyte of what follows the box.
constexpr uint32_t KBOX_BYTES = (128 + 8) * 128;
constexpr uint32_t KBUF_BYTES = 2 * KBOX_BYTES;
// TMEM columns: P (144 fp32 columns: the scores and, in column 128, phi(q) . z_prev), O and S (128 each); phi(Q) as
// packed bf16 pairs (64 columns); a 16-column block whose first column is z.  phi(Q) is the A operand of two products and goes from the registers
// that computed it straight to TMEM, so that the Q buffer in shared memory is free for the next tile as soon as it
// has been read.  The masked P goes back as packed bf16 pairs
// into the columns its own fp32 values came from: each thread overwrites only columns of its own row that it has
// already read (row r, tokens 64 hf + 32 qq ... + 31 -> columns 64 hf + 16 qq ... + 15).
constexpr uint32_t P_COL = 0, QZ_COL = 128, O_COL = 144, S_COL = 272, Z_COL = S_COL + 128, FQ_COL = 416 /* 64 columns */,
                   TMEM_COLS = 512;

// Shared-memory map (offsets from a 1024-byte aligned base).  The boxes of the two V buffers lie so that the block of
// ones that extends V to [V | 1] is the third box of both: buffer 0 in steps of one box, buffer 1 in steps of three, with
// Q in between.  [S | z] += phi(K)^T [V | 1] is then one product of 144 columns.  (As a product of its own, 16 columns
// wide, the extension cost as many cycles of the tensor cores as any: they take ~75 per instruction from 16 columns to
// 128, and every one of them reads phi(K) again: 1030 cycles per tile for the two, 616 for the one.)
constexpr uint32_t OFF_S = 0, OFF_K0 = TILE_BYTES, OFF_K1 = OFF_K0 + KBUF_BYTES, OFF_VQ = OFF_K1 + KBUF_BYTES,
                   OFF_Q = OFF_VQ + BOX_BYTES, OFF_ONES = OFF_VQ + 6 * BOX_BYTES;
static_assert(OFF_VQ % 1024 == 0, "swizzled boxes");
__host__ __device__ constexpr uint32_t vstep(uint32_t par) { return par ? 3 * BOX_BYTES : BOX_BYTES; }   // between a buffer's boxes
__host__ __device__ constexpr uint32_t vbox(uint32_t par, uint32_t half) {
  return OFF_VQ + (par ? 0u : 4 * BOX_BYTES) + half * vstep(par);
}
// The ones: a 128-byte-swizzled box of 128 rows of which the first 16 columns count (z3), or, where the taps of a long
// window leave no room for that, a block of 16 unswizzled columns (a product of its own, columns S_COL + 128 ...).
__host__ __device__ constexpr uint32_t ones_bytes(bool z3) { return z3 ? BOX_BYTES : 4096u; }
// [2][2][128] fp32: halves of the denominator of tile n in slot n & 1
__host__ __device__ constexpr uint32_t off_den(bool z3) { return OFF_ONES + ones_bytes(z3); }
__host__ __device__ constexpr uint32_t off_small(bool z3) { return off_den(z3) + 2048; }

struct Small {
  unsigned long long bars[25];
  uint32_t tmem_base;
  int abort;
};
// full_*: TMA landed.  PHI / PDONE / SB: arrivals of group A.  EPI0 / EPI1: arrivals of group B (the accumulator
// has been read; tiles alternate between the two).
// STAGED0 / STAGED1: group B has written a tile's outputs into that V buffer (the control lane stores them).
// MMA_P / MMA_S / MMA_Q / MMA_O: tcgen05.commit after P; after [S|z] += phi(K)^T [V|1] (K buffer free);
// after O = phi(Q) S_prev; after O += P V (MMA_O0 / MMA_O1, tiles alternate).
// A barrier that one role waits on while another role can run a tile ahead exists once per tile parity, so that a
// waiter is never more than one phase behind.
enum { B_FULL_K0 = 0, B_FULL_V0 = 1, B_FULL_V1 = 2, B_MMA_P = 3, B_MMA_S0 = 4, B_MMA_O0 = 5, B_MMA_O1 = 6, B_PHI = 7,
       B_PDONE = 8, B_SB = 9, B_EPI0 = 10, B_EPI1 = 11, B_MMA_Q = 12, B_FULL_Q = 13, B_FULL_K1 = 14, B_STAGED0 = 15,
       B_STAGED1 = 16, B_HALO0 = 17, B_HALO1 = 18, B_MMA_S1 = 19,
       B_MMA_L = 20 /* the scores against earlier groups of the tile */, 
       B_ST_PHI0 = 21, B_ST_PHI1 = 22, B_ST_MMA0 = 23, B_ST_MMA1 = 24 /* the state pass */, kNumBars = 25 };
static_assert(kNumBars <= 25 && sizeof(Small) == 208, "Small::bars");

__host__ __device__ constexpr uint32_t off_w(bool z3) { return off_small(z3) + (uint32_t)((sizeof(Small) + 15) / 16 * 16); }
// Short windows: nine halo buffers, rows of v that lie before 32 rows of a tile, for the convolution.  Buffers 0-2: the
// rows before tile n in n % 3; 3-8: the rows before rows 32, 64 and 96 of a tile, by the tile's parity.  Rows lie as in a
// V box (64 channels each, 128-byte swizzle; the row number counted back from the 32 rows: -1, -2, ...).
__host__ __device__ inline uint32_t off_halo(int W) { return (off_w(true) + (uint32_t)W * D * 4 + 127u) & ~127u; }
__host__ __device__ inline uint32_t halo_bytes(int W) { return (uint32_t)(W - 1) * 256u; }
__device__ __forceinline__ uint32_t halo_at(int i, int c16, int W) {   // row i (0 = oldest), 16-byte piece c16 of 16
  return (uint32_t)(c16 >> 3) * (uint32_t)(W - 1) * 128u + (uint32_t)i * 128u + (uint32_t)(((c16 & 7) ^ ((i - (W - 1)) & 7)) << 4);
}
__host__ __device__ inline uint32_t smem_bytes(int W) { return off_halo(W) + 9u * halo_bytes(W) + 1024; }
// The three-branch mode keeps 4 KB more behind the halo rows: z before the tile as fp32 [128], the halves of
// phi(q) . z [2][128], and each half-row's running maximum and sum of the softmax [2][128] x 2.
constexpr uint32_t kGrpScratch = 4096;
// The epilogue for longer tap windows ("long" below) keeps the taps padded with zeros to whole groups of 8 and ONE
// halo buffer, updated in place, of as many rows as the padded taps reach back (the rows before the window stay 0).
constexpr uint32_t kMaxSmem = 227u * 1024u;
__host__ __device__ inline uint32_t long_taps(int W) { return ((uint32_t)W + 7u) & ~7u; }
__host__ __device__ inline bool z3_long(int W, bool grp) {
  return off_w(true) + long_taps(W) * D * 4 + (long_taps(W) - 1) * D * 2 + 1024 + (grp ? kGrpScratch + 16u : 0u) <= kMaxSmem;
}
__host__ __device__ inline uint32_t off_halo_long(int W, bool grp) { return off_w(z3_long(W, grp)) + long_taps(W) * D * 4; }
__host__ __device__ inline uint32_t smem_bytes_long(int W, bool grp) { return off_halo_long(W, grp) + (long_taps(W) - 1) * D * 2 + 1024; }
__host__ __device__ inline uint32_t off_grp(int W, bool lng) {
  return ((lng ? smem_bytes_long(W, true) : smem_bytes(W)) - 1024 + 15u) & ~15u;
}
__host__ __device__ inline uint32_t smem_bytes_grp(int W, bool lng) { return off_grp(W, lng) + kGrpScratch + 1024; }
// Which windows take the long epilogue: above 5 taps the short one's nine halo buffers no longer fit (6 taps: 235 008 bytes
// of shared memory, kMaxSmem is 232 448).  The three-branch mode compiles the short epilogue for 3 taps only.
inline bool long_epilogue(int W, bool grouped = false) { return grouped ? W != 3 : W > 5; }

// ---- PTX wrappers ------------------------------------------------------------------------
__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint32_t bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void mbar_inval(uint32_t bar) { asm volatile("mbarrier.inval.shared::cta.b64 [%0];" ::"r"(bar) : "memory"); }
__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire;" ::: "memory"); }
__device__ __forceinline__ void fence_proxy_async() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void sync_group_b() { asm volatile("bar.sync 2, 256;" ::: "memory"); }
__device__ __forceinline__ void sync_group_a() { asm volatile("bar.sync 5, 256;" ::: "memory"); }
template <int N> __device__ __forceinline__ void regs_up() { asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(N)); }
template <int N> __device__ __forceinline__ void regs_down() { asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(N)); }
__device__ __forceinline__ float ex2(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
__device__ __forceinline__ void tma_load(uint32_t dst, const CUtensorMap* map, int x, int y, int z, uint32_t bar) {
  asm volatile(
      "cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4}], [%5];"
      ::"r"(dst), "l"(map), "r"(x), "r"(y), "r"(z), "r"(bar)
      : "memory");
}
__device__ __forceinline__ void tma_store(const CUtensorMap* map, int x, int y, int z, uint32_t src) {
  asm volatile("cp.async.bulk.tensor.3d.global.shared::cta.bulk_group [%0, {%1, %2, %3}], [%4];" ::"l"(map), "r"(x),
               "r"(y), "r"(z), "r"(src)
               : "memory");
}
__device__ __forceinline__ void tma_commit() { asm volatile("cp.async.bulk.commit_group;" ::: "memory"); }
__device__ __forceinline__ void tma_wait_read() { asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory"); }
__device__ __forceinline__ void tma_wait_all() { asm volatile("cp.async.bulk.wait_group 0;" ::: "memory"); }

__device__ __forceinline__ void mma_bf16(uint32_t d_tmem, uint64_t a_desc, uint64_t b_desc, uint32_t idesc, bool acc) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}"
      ::"r"(d_tmem), "l"(a_desc), "l"(b_desc), "r"(idesc), "r"((uint32_t)acc)
      : "memory");
}
// The same with the A operand read from TMEM (rows in lanes, two bf16 per 32-bit column).
__device__ __forceinline__ void mma_bf16_ts(uint32_t d_tmem, uint32_t a_tmem, uint64_t b_desc, uint32_t idesc, bool acc) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n\t}"
      ::"r"(d_tmem), "r"(a_tmem), "l"(b_desc), "r"(idesc), "r"((uint32_t)acc)
      : "memory");
}
// ... and with the first `off` lanes (0, 32, 64 or 96) of the accumulator left as they are.
__device__ __forceinline__ void mma_bf16_ts_below(uint32_t d_tmem, uint32_t a_tmem, uint64_t b_desc, uint32_t idesc, bool acc, int off) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, {%5, %6, %7, %8}, p;\n\t}"
      ::"r"(d_tmem), "r"(a_tmem), "l"(b_desc), "r"(idesc), "r"((uint32_t)acc), "r"(off > 0 ? ~0u : 0u), "r"(off > 32 ? ~0u : 0u),
        "r"(off > 64 ? ~0u : 0u), "r"(0u)
      : "memory");
}
__device__ __forceinline__ void mma_commit(uint32_t bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}

#define LA_TMEM_LD32(taddr, r)                                                                                   \
  asm volatile(                                                                                                  \
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 "                                                                  \
      "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "                                  \
      "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"                  \
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),          \
        "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]),    \
        "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]),  \
        "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])   \
      : "r"(taddr)                                                                                               \
      : "memory")

#define LA_TMEM_ST32(taddr, r)                                                                                   \
  asm volatile(                                                                                                  \
      "tcgen05.st.sync.aligned.32x32b.x32.b32 [%0], "                                                            \
      "{%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, %16, "                                 \
      "%17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31, %32};"                         \
      ::"r"(taddr), "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]),      \
        "r"(r[8]), "r"(r[9]), "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15]),            \
        "r"(r[16]), "r"(r[17]), "r"(r[18]), "r"(r[19]), "r"(r[20]), "r"(r[21]), "r"(r[22]), "r"(r[23]),          \
        "r"(r[24]), "r"(r[25]), "r"(r[26]), "r"(r[27]), "r"(r[28]), "r"(r[29]), "r"(r[30]), "r"(r[31])           \
      : "memory")

// Fragments of 8 rows x 8 columns: 16 TMEM lanes x 8 G columns at once; register 4 g + 2 i + e of lane l holds row
// (l >> 2) + 8 i, column 8 g + 2 (l & 3) + e.  Four lanes then hold 32 consecutive bytes of an fp32 row, one sector of
// global memory: the layout in which a state moves between TMEM and HBM (with a row per lane every access touched 32
// cache lines, 16 bytes each: 3 us to write one 64 KB state, as long as a tile takes).
#define LA_TMEM_LD_FRAG8(taddr, r)                                                                               \
  asm volatile(                                                                                                  \
      "tcgen05.ld.sync.aligned.16x256b.x8.b32 "                                                                  \
      "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "                                  \
      "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"                  \
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),          \
        "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]),    \
        "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]),  \
        "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])   \
      : "r"(taddr)                                                                                               \
      : "memory")
#define LA_TMEM_ST_FRAG4(taddr, r)                                                                               \
  asm volatile(                                                                                                  \
      "tcgen05.st.sync.aligned.16x256b.x4.b32 [%0], "                                                            \
      "{%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, %16};"                                 \
      ::"r"(taddr), "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]),      \
        "r"(r[8]), "r"(r[9]), "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15])             \
      : "memory")
#define LA_TMEM_LD_FRAG4(taddr, r)                                                                               \
  asm volatile(                                                                                                  \
      "tcgen05.ld.sync.aligned.16x256b.x4.b32 "                                                                  \
      "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"                           \
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),          \
        "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])     \
      : "r"(taddr)                                                                                               \
      : "memory")
// Global side of a fragment of 64 columns; `p` is this lane's first element (row l >> 2, column 2 (l & 3)) of a [..][128]
// matrix.
__device__ __forceinline__ void frag_load(const float* p, uint32_t (&r)[32]) {
#pragma unroll
  for (int g = 0; g < 8; ++g)
#pragma unroll
    for (int i = 0; i < 2; ++i) {
      const float2 x = *reinterpret_cast<const float2*>(p + i * 8 * D + 8 * g);
      r[4 * g + 2 * i] = __float_as_uint(x.x);
      r[4 * g + 2 * i + 1] = __float_as_uint(x.y);
    }
}
__device__ __forceinline__ void frag_add(uint32_t (&r)[32], const uint32_t (&x)[32]) {
#pragma unroll
  for (int e = 0; e < 32; ++e) r[e] = __float_as_uint(__uint_as_float(r[e]) + __uint_as_float(x[e]));
}
__device__ __forceinline__ void frag_store(float* p, const uint32_t (&r)[32]) {
#pragma unroll
  for (int g = 0; g < 8; ++g)
#pragma unroll
    for (int i = 0; i < 2; ++i)
      *reinterpret_cast<float2*>(p + i * 8 * D + 8 * g) =
          make_float2(__uint_as_float(r[4 * g + 2 * i]), __uint_as_float(r[4 * g + 2 * i + 1]));
}
// 8 x 8 matrices of bf16 between shared memory and the same fragments: lane l names the 16-byte row l & 7 of matrix l >> 3.
__device__ __forceinline__ void ldmatrix4(uint32_t a, uint32_t (&r)[4]) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0, %1, %2, %3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"(a)
               : "memory");
}
__device__ __forceinline__ void stmatrix4(uint32_t a, const uint32_t (&r)[4]) {
  asm volatile("stmatrix.sync.aligned.m8n8.x4.shared.b16 [%0], {%1, %2, %3, %4};" ::"r"(a), "r"(r[0]), "r"(r[1]), "r"(r[2]),
               "r"(r[3])
               : "memory");
}

__device__ __forceinline__ uint32_t tmem_ld1(uint32_t taddr) {
  uint32_t v;
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x1.b32 {%0}, [%1];" : "=r"(v) : "r"(taddr) : "memory");
  return v;
}
__device__ __forceinline__ void tmem_st1(uint32_t taddr, uint32_t v) {
  asm volatile("tcgen05.st.sync.aligned.32x32b.x1.b32 [%0], {%1};" ::"r"(taddr), "r"(v) : "memory");
}
#define LA_TMEM_ST16(taddr, r)                                                                                   \
  asm volatile(                                                                                                  \
      "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], "                                                            \
      "{%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, %16};"                                 \
      ::"r"(taddr), "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]),      \
        "r"(r[8]), "r"(r[9]), "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15])             \
      : "memory")

#define LA_TMEM_LD16(taddr, r)                                                                                   \
  asm volatile(                                                                                                  \
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 "                                                                  \
      "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"                           \
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),          \
        "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])     \
      : "r"(taddr)                                                                                               \
      : "memory")
__device__ __forceinline__ void tmem_st8(uint32_t taddr, const uint32_t* r) {
  asm volatile("tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"r"(taddr), "r"(r[0]),
               "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7])
               : "memory");
}

__device__ __forceinline__ void tmem_wait_ld() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }
__device__ __forceinline__ void tmem_wait_st() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }

// ---- descriptors ----------------------------------------------------------------------------
// Shared-memory matrix descriptor: start address, leading and stride byte offsets (16-byte units),
// descriptor version 1, layout type (2 = 128-byte swizzle, 0 = no swizzle).
__device__ __forceinline__ uint64_t smem_desc(uint32_t addr, uint32_t lbo_bytes, uint32_t sbo_bytes, uint32_t layout) {
  return (uint64_t)((addr >> 4) & 0x3FFFu) | ((uint64_t)((lbo_bytes >> 4) & 0x3FFFu) << 16) |
         ((uint64_t)((sbo_bytes >> 4) & 0x3FFFu) << 32) | (1ull << 46) | ((uint64_t)layout << 61);
}
// Operand whose contraction index runs along the 128-byte rows (rows = M or N): step ks covers 16 elements.
__device__ __forceinline__ uint64_t desc_kmajor(uint32_t tile, int ks) {
  return smem_desc(tile + (uint32_t)(ks >> 2) * BOX_BYTES + (uint32_t)(ks & 3) * 32u, 16u, 1024u, 2u);
}
// Operand whose contraction index runs along the tile rows (rows = K, 128-byte rows hold M or N): step ks
// covers 16 rows; the two 64-element column boxes are BOX_BYTES apart.
__device__ __forceinline__ uint64_t desc_mnmajor(uint32_t tile, int ks) {
  return smem_desc(tile + (uint32_t)ks * 2048u, BOX_BYTES, 1024u, 2u);
}
// The 16-column extensions ([128 rows = K] x [16 = N], no swizzle): 8 x 8 cores of 128 bytes, the two cores of
// one 8-row group side by side (stride 128 B along N), 8-row groups 256 B apart (stride along K).
__device__ __forceinline__ uint64_t desc_ext(uint32_t tile, int ks) {
  return smem_desc(tile + (uint32_t)ks * 512u, 256u, 128u, 0u);
}
__device__ __forceinline__ uint32_t ext_offset(int k, int n) {   // byte offset of element (k, n) in such a block
  return (uint32_t)(k >> 3) * 256u + (uint32_t)(n >> 3) * 128u + (uint32_t)(k & 7) * 16u + (uint32_t)(n & 7) * 2u;
}
// The same descriptors split into their two 32-bit words: the steps of a product differ only in the start-address
// field of the low word (by a constant, and the field cannot overflow below 256 KB), so the issuing lane forms the
// words of step 0 once per tile and adds a constant per step.
__device__ __forceinline__ uint32_t desc_lo(uint32_t addr, uint32_t lbo_bytes) {
  return ((addr >> 4) & 0x3FFFu) | (((lbo_bytes >> 4) & 0x3FFFu) << 16);
}
constexpr uint32_t kDescHiSw128 = ((1024u >> 4) & 0x3FFFu) | (1u << 14) | (2u << 29);   // SBO 1024, version 1, 128-byte swizzle
__host__ __device__ constexpr uint32_t kstep_kmajor(int ks, uint32_t box = BOX_BYTES) { return ((uint32_t)(ks >> 2) * box + (uint32_t)(ks & 3) * 32u) >> 4; }
__host__ __device__ constexpr uint32_t kstep_mnmajor(int ks) { return ((uint32_t)ks * 2048u) >> 4; }
__device__ __forceinline__ uint64_t desc64(uint32_t lo) { return ((uint64_t)kDescHiSw128 << 32) | lo; }
// Instruction descriptor: fp32 accumulate, bf16 x bf16, M = 128, N = n.
__host__ __device__ constexpr uint32_t idesc(bool a_mn, bool b_mn, uint32_t n) {
  return (1u << 4) | (1u << 7) | (1u << 10) | ((a_mn ? 1u : 0u) << 15) | ((b_mn ? 1u : 0u) << 16) |
         ((n >> 3) << 17) | ((128u >> 4) << 24);
}

// ---- bf16 packing ------------------------------------------------------------------------------
__device__ __forceinline__ uint32_t pack2(float a, float b) {
  __nv_bfloat162 h = __floats2bfloat162_rn(a, b);
  return *reinterpret_cast<uint32_t*>(&h);
}
__device__ __forceinline__ float lo_f(uint32_t u) { return __uint_as_float(u << 16); }
__device__ __forceinline__ float hi_f(uint32_t u) { return __uint_as_float(u & 0xffff0000u); }

// phi on two packed bf16 values, entirely in packed arithmetic.  elu+1: x + 1 where x > 0 (one correctly
// rounded bf16 addition), 2^(x log2 e) elsewhere; the two are merged with a lane mask.  The exponent argument is
// formed by one fused multiply (x * log2e_hi + x * log2e_lo would not help: the product is rounded to bf16
// either way), so exp(x) carries a relative error of about |x| 2^-9 on top of the bf16 rounding of the result --
// below one bf16 ulp for |x| < 1, and in absolute terms largest where exp(x) is close to 1.  ReLU: packed max.
template <int PHI> __device__ __forceinline__ uint32_t phi2(uint32_t u) {
  if (PHI == LA_PHI_ELU1) {
    uint32_t y, e, xp1, mask;
    asm("mul.rn.bf16x2 %0, %1, %2;" : "=r"(y) : "r"(u), "r"(0x3fb93fb9u));        // log2(e) = 1.4453 in bf16
    asm("ex2.approx.ftz.bf16x2 %0, %1;" : "=r"(e) : "r"(y));
    asm("add.rn.bf16x2 %0, %1, %2;" : "=r"(xp1) : "r"(u), "r"(0x3f803f80u));
    asm("set.gt.u32.bf16x2 %0, %1, %2;" : "=r"(mask) : "r"(u), "r"(0u));
    return (xp1 & mask) | (e & ~mask);
  }
  uint32_t r;
  asm("max.bf16x2 %0, %1, %2;" : "=r"(r) : "r"(u), "r"(0u));
  return r;
}
template <int PHI> __device__ __forceinline__ uint4 phi8(uint4 u) {
  return make_uint4(phi2<PHI>(u.x), phi2<PHI>(u.y), phi2<PHI>(u.z), phi2<PHI>(u.w));
}

// Byte offset of 16-byte chunk `cc` (0..7) of row `row` inside one 128-byte-swizzled box.
__device__ __forceinline__ uint32_t swz(int row, int cc) { return (uint32_t)row * 128u + (uint32_t)((cc ^ (row & 7)) << 4); }

// ---- the kernel ------------------------------------------------------------------------------------
// (Two channels per packed fp32 multiply-add: each half is the IEEE fused multiply-add of the scalar instruction.)
__device__ __forceinline__ float2 bf2(uint32_t u) { return make_float2(lo_f(u), hi_f(u)); }
// Long-window epilogue: one thread owns a pair of channels and 32 consecutive rows of the tile, in two blocks of 16.
// conv_block adds one group of 8 taps to the 16 sums of a block: the 23 rows of v that those taps reach are each read once,
// as one packed pair, and feed up to 8 of the sums.  (Blocks of 8 rows read and unpack 15 rows for half as many sums: 32 taps, 128
// chains of 2048 tokens, 139.4 us; 126.4 so.)
// The rows come from the V buffer (pg[k]: the thread's column, in the swizzle of rows = k mod 8, 8 g rows before the block's
// first), so that every load is one instruction with an immediate offset; HALO: the first nh of them from the halo column
// (hq: the first of the 23).  Two copies of the loop and not one per nh, of which there are four: it has to stay in the
// instruction cache (segments of 4 tiles, 9 taps: 40.4 us in blocks of 8, 44.1 with four copies, 40.1 with two).
template <int I, int N, typename F>
__device__ __forceinline__ void static_for(F&& f) {           // f(integral_constant<int, I>) ... for I, I + 1, ..., N - 1
  if constexpr (I < N) {
    f(std::integral_constant<int, I>{});
    static_for<I + 1, N>(f);
  }
}
// (Shared-memory addresses as 32-bit numbers and explicit ld.shared / st.shared: one register per address.)
__device__ __forceinline__ uint32_t lds32(uint32_t a) {
  uint32_t v;
  asm volatile("ld.shared.u32 %0, [%1];" : "=r"(v) : "r"(a));
  return v;
}
__device__ __forceinline__ float2 lds_f2(uint32_t a) {
  float2 v;
  asm volatile("ld.shared.v2.f32 {%0, %1}, [%2];" : "=f"(v.x), "=f"(v.y) : "r"(a));
  return v;
}
__device__ __forceinline__ void sts32(uint32_t a, uint32_t v) { asm volatile("st.shared.u32 [%0], %1;" ::"r"(a), "r"(v) : "memory"); }
template <bool HALO>
__device__ __forceinline__ void conv_block(float2 (&acc)[16], uint32_t wtap, const uint32_t (&pg)[8], uint32_t hq, int nh) {
  float2 wg[8];
  static_for<0, 8>([&](auto tc_) {
    constexpr int t = decltype(tc_)::value;
    wg[t] = lds_f2(wtap + t * (D * 4));
  });
  static_for<0, 23>([&](auto ic) {
    constexpr int i = decltype(ic)::value;
    const uint32_t a = pg[(i + 1) & 7] + (i - 7) * 128, u = lds32(HALO && i < nh ? hq + i * (D * 2) : a);
    const float2 x = bf2(u);
    static_for<0, 8>([&](auto tc_) {
      constexpr int tau = decltype(tc_)::value;   // tap (within the group) that links input row i to sum jj
      constexpr int jj = i - 7 + tau;
      if constexpr (jj >= 0 && jj < 16) acc[jj] = __ffma2_rn(wg[tau], x, acc[jj]);
    });
  });
}
// All tap groups of block blk (rows 16 blk ... 16 blk + 15 of the thread), then the sums are added to the attention
// term that waits in the output tile.  first: the thread owns the first 32 rows of the tile (rows before them
// come from the halo, hend = the halo column just past its last row).
__device__ __forceinline__ void conv_rows(int blk, bool first, uint32_t wcol, const uint32_t (&pv)[8], uint32_t sthr, int cc,
                                          uint32_t hend, int ngroups) {
  float2 acc[16];
#pragma unroll
  for (int jj = 0; jj < 16; ++jj) acc[jj] = make_float2(0.f, 0.f);
#pragma unroll 1
  for (int g = 0; g < ngroups; ++g) {
    const uint32_t wtap = wcol + g * (8 * D * 4), hq = hend + (16 * blk - 8 * g - 7) * (D * 2);
    const int m = first ? g - 2 * blk : -1;
    uint32_t pg[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) pg[k] = pv[k] + (2 * blk - g) * 1024;
    if (m < 0) conv_block<false>(acc, wtap, pg, hq, 0);
    else conv_block<true>(acc, wtap, pg, hq, 8 * m + 7);
  }
  sthr += blk * 2048;
#pragma unroll
  for (int j0 = 0; j0 < 16; j0 += 8) {
    uint32_t lav[8];                              // the attention terms of 8 rows, all loads in flight at once
#pragma unroll
    for (int jj = 0; jj < 8; ++jj) lav[jj] = lds32(sthr + (j0 + jj) * 128 + ((cc ^ jj) << 4));
#pragma unroll
    for (int jj = 0; jj < 8; ++jj) {
      const float2 la = bf2(lav[jj]);
      sts32(sthr + (j0 + jj) * 128 + ((cc ^ jj) << 4), pack2(acc[j0 + jj].x + la.x, acc[j0 + jj].y + la.y));
    }
  }
}

enum { ALL_V = 0, MIXED = 1, ALL_H = 2 };
template <int KIND>
__device__ __forceinline__ void conv_block8(float2 (&acc)[8], uint32_t wtap, const uint32_t (&pg)[8], uint32_t hq) {
  float2 wg[8];
  static_for<0, 8>([&](auto tc_) {
    constexpr int t = decltype(tc_)::value;
    wg[t] = lds_f2(wtap + t * (D * 4));
  });
  static_for<0, 15>([&](auto ic) {
    constexpr int i = decltype(ic)::value;
    uint32_t u;
    if constexpr (KIND == ALL_V) {
      u = lds32(pg[(i + 1) & 7] + (i - 7) * 128);
    } else if constexpr (KIND == ALL_H || i < 7) {
      u = lds32(hq + i * (D * 2));
    } else {
      u = lds32(pg[i - 7] + (i - 7) * 128);
    }
    const float2 x = bf2(u);
    static_for<0, 8>([&](auto tc_) {
      constexpr int tau = decltype(tc_)::value;   // tap (within the group) that links input row i to sum jj
      constexpr int jj = i - 7 + tau;
      if constexpr (jj >= 0 && jj < 8) acc[jj] = __ffma2_rn(wg[tau], x, acc[jj]);
    });
  });
}
// The same in blocks of 8 rows, whose code is half as long: for windows of one group of taps, which is gone through once per block
// (segments of 4 tiles, 6 taps: 36.1 us, 38.7 in blocks of 16; 128 whole chains of 2048 tokens 84.4 and 85.3), and for the
// three-branch mode (16 taps, groups of 64: 52.7 and 55.6).
// conv_block8: rows -7 ... 7 of a block all from the V buffer (ALL_V), all from the halo (ALL_H), or the negative ones (MIXED).
// All tap groups of block blk (rows 8 blk ... 8 blk + 7 of the thread), then the sums are added to the attention
// term that waits in the output tile.  first: the thread owns the first 32 rows of the tile (rows before them
// come from the halo, hend = the halo column just past its last row).
__device__ __forceinline__ void conv_rows8(int blk, bool first, uint32_t wcol, const uint32_t (&pv)[8], uint32_t sthr, int cc,
                                          uint32_t hend, int ngroups) {
  float2 acc[8];
#pragma unroll
  for (int jj = 0; jj < 8; ++jj) acc[jj] = make_float2(0.f, 0.f);
#pragma unroll 1
  for (int g = 0; g < ngroups; ++g) {
    const uint32_t wtap = wcol + g * (8 * D * 4);
    if (!first || g < blk) {
      uint32_t pg[8];
#pragma unroll
      for (int k = 0; k < 8; ++k) pg[k] = pv[k] + (blk - g) * 1024;
      conv_block8<ALL_V>(acc, wtap, pg, 0u);
    } else if (g == blk) {
      conv_block8<MIXED>(acc, wtap, pv, hend - 7 * (D * 2));
    } else {
      conv_block8<ALL_H>(acc, wtap, pv, hend + (8 * (blk - g) - 7) * (D * 2));
    }
  }
  sthr += blk * 1024;
  uint32_t lav[8];                                // the attention terms of the 8 rows, all loads in flight at once
#pragma unroll
  for (int jj = 0; jj < 8; ++jj) lav[jj] = lds32(sthr + jj * 128 + ((cc ^ jj) << 4));
#pragma unroll
  for (int jj = 0; jj < 8; ++jj) {
    const float2 la = bf2(lav[jj]);
    sts32(sthr + jj * 128 + ((cc ^ jj) << 4), pack2(acc[jj].x + la.x, acc[jj].y + la.y));
  }
}

__device__ __forceinline__ uint4 pack8(const uint32_t* v) {
  return make_uint4(pack2(__uint_as_float(v[0]), __uint_as_float(v[1])), pack2(__uint_as_float(v[2]), __uint_as_float(v[3])),
                    pack2(__uint_as_float(v[4]), __uint_as_float(v[5])), pack2(__uint_as_float(v[6]), __uint_as_float(v[7])));
}

// GM > 0 (GRP): the three-branch block of Sec. 4.1.  The score product runs on the raw q and k and its rows go through a
// causal softmax inside their group (left branch); the products with the state of the earlier tiles are the
// group-exclusive linear attention (middle branch); both land in one accumulator, the probabilities pre-scaled by
// (phi(q).z + eps) / alpha so that one row factor finishes both.
// GM = 1: one group per tile (partly filled where the group is shorter than 128), no intra-tile linear term.
// GM = 2 (MULTI): 128 / gsz groups of gsz = 32 or 64 tokens per tile.  A row then also meets the earlier groups of its
// tile, linearly: a product per group, phi(Q) with phi(K) of that group, puts those scores in the place of the raw ones
// that nobody needs (the accumulator's other lanes are masked off), and they join P unscaled, as two bf16 numbers each:
// the rounding of a score, unlike that of an entry of S, is not averaged over the 128 features (rounded once, they left
// the global branch of values that cancel 30 times further from its exact value than the state's copy does).  P of 16
// tokens c ... c + 15 takes the place of their fp32 scores: columns c ... c + 7, and c + 8 ... c + 15 for what the rounding
// of the linear ones left over, so that every thread overwrites only what it has read itself.  (One partly filled tile
// per group of 64 took 200 us on 128 chains of 2048 tokens, as long per tile as a full one.)
template <int PHI, int WT, int GM = 0>
__global__ void __launch_bounds__(kThreads, 1)
prefill_tc_kernel(const __grid_constant__ CUtensorMap mq, const __grid_constant__ CUtensorMap mk,
                  const __grid_constant__ CUtensorMap mv, const __grid_constant__ CUtensorMap mo,
                  const float* __restrict__ w, float* __restrict__ S, float* __restrict__ z,
                  __nv_bfloat16* __restrict__ win, int64_t* __restrict__ pos,
                  int* status, int H, int Ttot, int W, float eps, int init, int nseg,
                  int seg_len, float* S_seg, float* z_seg,
                  const __nv_bfloat16* __restrict__ win_seg, int prefixed, int fused, const __nv_bfloat16* __restrict__ vg,
                  int v_chain, int v_seg, float alpha,
                  float sm_scale, int tstep, int gsz, int early) {
  extern __shared__ unsigned char smem_dyn[];
  // (an offset into the array rather than an integer cast: the compiler then knows that these are shared-memory
  // addresses: 32-bit arithmetic, ld.shared / st.shared)
  unsigned char* smem = smem_dyn + ((1024u - (smem_u32(smem_dyn) & 1023u)) & 1023u);
  const uint32_t sbase = smem_u32(smem);
  constexpr bool GRP = GM > 0, MULTI = GM == 2;
  constexpr bool LONG = WT < 0;                  // the epilogue for longer tap windows
  // One group of 8 taps (WT = -1) and more (-2) are kernels of their own: with both forms of the tap loop in one, 32 chains of 1700
  // tokens, 9 to 16 taps, took 1 % longer than with either alone.  (Three-branch mode: one form, -1.)
  constexpr bool ONE8 = WT == -1 && !GRP;
  // The exact layer with a short window keeps its loops rolled: all roles' code of one tile has to stay in the SM's instruction
  // cache.  (Unrolled, 23 KB of it came anew with every tile from the cache that a GPC shares, and two of a scheduler's five
  // warps waited for instructions on average, 0.6 of them now: 128 chains of 2048 tokens, 3 taps, in runs too short for the power
  // limit 66.8 us before, 61.6 since; back to back, where the clock gives way, 72.1 and 71.5.  32 chains of 1700 tokens 37.4 and
  // 35.2.)  Not the three-branch mode, whose phi lies on the longest chain of a tile (groups of 64:
  // 95 us, 104 rolled), nor long windows, whose tap sums leave little of the wait (32 taps: 127.2 us, 128.9 rolled).
  // (phi(K) and the epilogue only beside an elu + 1: a ReLU has little code, and the loads that a rolled loop waits for show.  ReLU, 1 to 4
  // taps: 128 and 256 chains of 1000 or 2048 tokens 0.4-0.9 % faster unrolled, 32 chains of 1700 2 %, one tile 0.5-1 %.)
  constexpr bool kRoll = !LONG && !GRP, kRollE = kRoll && PHI == LA_PHI_ELU1;
  // Who copies the state between two tiles: group B has the time beside an elu + 1 (which keeps group A busy), group A beside
  // a ReLU or a long window (which keeps group B busy).
  constexpr bool SNAP_A = LONG || (PHI == LA_PHI_RELU && !GRP);
  // Of the 128 rows of phi(K) group B takes the last 16 KB, beside an elu + 1 with a short window: group A's loop (phi(Q),
  // phi(K), mask) is the longest there, and group B had 2 K of a tile's 5.9 K cycles to spare.  (128 chains of 2048 tokens,
  // 3 taps: 71 us with none, 65.4 with 2, 64.6 with 3, 65.8 with 4.)
  constexpr int KB = SNAP_A || GRP ? 0 : 3;
  // Long windows and the three-branch mode: registers per thread once the roles have traded theirs.  256 threads of group
  // A, 256 of group B and 128 others were launched with 96 each: 2 kRegsA + 2 kRegsB + 64 = 5 x 96.
  constexpr bool TRADE = LONG || GRP;
  // (Group A of the ReLU holds fewer values and fits in 88; group B spills with 112 there and not with 120: 32 taps, 128
  // chains of 2048 tokens 135.2 -> 133.2 us, 8 taps 80.1 -> 77.8.  The elu + 1 with 88: 139.5 -> 141.2.)
  constexpr int kRegsA = LONG && !GRP && PHI == LA_PHI_RELU ? 88 : LONG && !MULTI ? 96 : LONG ? 104 : 112;
  constexpr int kRegsB = 208 - kRegsA;
  static_assert(kThreadsA == 256 && kThreadsB == 256 && kThreads == 640, "register split");
  // Whose waits are the tight ones (see mbar_wait).  Long windows, elu + 1: those of the issuing, copying and halo warps (means over 12
  // shapes: 6 to 8 taps 0.3-0.6 % faster, 9 to 32 taps 1.0-1.4 %; with ReLU 0.5-1.9 % slower from 9 taps on).
  // Three-branch mode, one group per tile: those of group A with 3 taps (54 shapes, groups of 33 to 128 tokens: 2-4 % faster), those of
  // group B otherwise (3-5 %; without, these kernels spill 20 bytes).  Groups that share a tile: nobody's (0-4 % slower).
  constexpr bool TIGHT_C = LONG && !GRP && PHI == LA_PHI_ELU1, TIGHT_A = GM == 1 && !LONG, TIGHT_B = GM == 1 && LONG;
  const bool z3 = LONG ? z3_long(W, GRP) : true; // z rides in the state update's product
  Small& sm = *reinterpret_cast<Small*>(smem + off_small(z3));
  float* wsm = reinterpret_cast<float*>(smem + off_w(z3));                     // [W][128] ([W up to a multiple of 8][128] if LONG)
  __nv_bfloat16* halo0 = reinterpret_cast<__nv_bfloat16*>(smem + (LONG ? off_halo_long(W, GRP) : off_halo(W)));
  volatile int* abort = &sm.abort;
  // three-branch mode only: z before the tile (fp32), the halves of phi(q) . z, the halves of the softmax statistics
  float* zs = reinterpret_cast<float*>(smem + off_grp(W, LONG));               // [128]
  float* dgh = zs + D;                                                         // [2][128]
  float2* mlh = reinterpret_cast<float2*>(dgh + 2 * D);                        // [2][128] (max, sum)
  const bool use_glob = GRP && alpha != 0.f;     // alpha = 0: the global branch is switched off altogether

  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  // A launch covers BH chains cut into nseg segments of seg_len tokens (nseg = 1: whole chains).  This block owns
  // tokens [y0, y0 + T) of chain bh.  Whole chains start from the caller's state, the segments sg > 0 of a chain that was
  // cut from the sums of the segments before them and from the values of v before them; only the last segment writes a
  // state, the caller's.  Where the sums come from:
  //   fused     the segments of a chain are one cluster: each block first forms its own segment's sums (the state pass),
  //             leaves them in the workspace, and after a barrier of the cluster adds up those before it;
  //   else      a launch of its own formed them (and left a copy of the caller's state for segment 0 in the last slot), and
  //             with `prefixed` another one added them up: slot sg - 1.
  // Either way the first segment's sums have the caller's state in them.
  const int bh = blockIdx.x / nseg, sg = blockIdx.x % nseg, h = bh % H;
  const int y0 = sg * seg_len, T = min(seg_len, Ttot - y0);
  const bool has_in = init || sg > 0, writes_state = sg == nseg - 1;
  const bool callers = nseg == 1 || (fused && sg == 0);   // the incoming state is the caller's
  const int nsum = sg > 0 && !prefixed ? sg : 1;          // how many parts it has
  const size_t slot = (size_t)bh * nseg + (fused ? 0 : sg == 0 ? nseg - 1 : prefixed ? sg - 1 : 0);
  const float *S_in = callers ? S + (size_t)bh * D * D : S_seg + slot * D * D, *z_in = callers ? z + (size_t)bh * D : z_seg + slot * D;
  // (the rows before segment sg: row bh * v_chain + sg * v_seg - (W - 1) ... of vg, which is v or holds copies of just these rows)
  const __nv_bfloat16* win_in = sg > 0 ? vg + ((size_t)bh * v_chain + sg * v_seg - (W - 1)) * D
                                       : (nseg > 1 && !fused ? win_seg : win) + (size_t)bh * (W - 1) * D;
  auto z_start = [&](int a) {
    float x = z_in[a];
    for (int j = 1; j < nsum; ++j) x += z_in[j * D + a];
    return x;
  };
  // tstep: tokens per tile, 128 except for three-branch groups shorter than that, which take one partly filled tile
  // each (the TMA boxes are then tstep rows high; the rows below hold zeros or values that the causal mask discards).
  const int nchunks = (T + tstep - 1) / tstep;
  const uint32_t tile_tx = (uint32_t)tstep * 256u;            // bytes a tile's two boxes bring
  const uint32_t bar0 = smem_u32(&sm.bars[0]);    // barrier i lives at bar0 + 8 i

  auto load_k = [&](int n) {                      // K / V of tile n into the buffers of its parity (one thread)
    const uint32_t kb = sbase + ((n & 1) ? OFF_K1 : OFF_K0), kbar = bar0 + 8u * ((n & 1) ? B_FULL_K1 : B_FULL_K0);
    mbar_expect_tx(kbar, tile_tx);
    tma_load(kb, &mk, 0, y0 + n * tstep, bh, kbar);
    tma_load(kb + KBOX_BYTES, &mk, 64, y0 + n * tstep, bh, kbar);
  };
  auto load_v = [&](int n) {
    const uint32_t vbar = bar0 + 8u * (B_FULL_V0 + (n & 1));
    mbar_expect_tx(vbar, tile_tx);
    tma_load(sbase + vbox(n & 1, 0), &mv, 0, y0 + n * tstep, bh, vbar);
    tma_load(sbase + vbox(n & 1, 1), &mv, 64, y0 + n * tstep, bh, vbar);
  };

  auto load_q0 = [&]() {
    mbar_expect_tx((bar0 + 8u * (B_FULL_Q)), tile_tx);
    tma_load(sbase + OFF_Q, &mq, 0, y0, bh, (bar0 + 8u * (B_FULL_Q)));
    tma_load(sbase + OFF_Q + BOX_BYTES, &mq, 64, y0, bh, (bar0 + 8u * (B_FULL_Q)));
  };

  // ---- set-up ----
  if (tid == kCopyWarp * 32) {
    mbar_init((bar0 + 8u * (B_FULL_K0)), 1);
    mbar_init((bar0 + 8u * (B_FULL_K1)), 1);
    mbar_init((bar0 + 8u * (B_FULL_Q)), 1);
    mbar_init((bar0 + 8u * (B_FULL_V0)), 1);
    mbar_init((bar0 + 8u * (B_FULL_V1)), 1);
    mbar_init((bar0 + 8u * (B_MMA_P)), 1);
    mbar_init((bar0 + 8u * (B_MMA_S0)), 1);
    mbar_init((bar0 + 8u * (B_MMA_S1)), 1);
    mbar_init((bar0 + 8u * (B_MMA_L)), 1);
    mbar_init((bar0 + 8u * (B_MMA_O0)), 1);
    mbar_init((bar0 + 8u * (B_MMA_O1)), 1);
    mbar_init((bar0 + 8u * (B_PHI)), kThreadsA);
    mbar_init((bar0 + 8u * (B_PDONE)), kThreadsA);
    mbar_init((bar0 + 8u * (B_SB)), SNAP_A ? kThreadsA : kThreadsB);
    mbar_init((bar0 + 8u * (B_EPI0)), kThreadsB);
    mbar_init((bar0 + 8u * (B_EPI1)), kThreadsB);
    mbar_init((bar0 + 8u * (B_MMA_Q)), 1);
    mbar_init((bar0 + 8u * (B_STAGED0)), kThreadsB);
    mbar_init((bar0 + 8u * (B_STAGED1)), kThreadsB);
    mbar_init((bar0 + 8u * (B_HALO0)), 32);
    mbar_init((bar0 + 8u * (B_HALO1)), 32);
    for (int i = 0; i < 2; ++i) {
      mbar_init((bar0 + 8u * (B_ST_MMA0 + i)), 1);
      mbar_init((bar0 + 8u * (B_ST_PHI0 + i)), kThreadsA + kThreadsB);
    }
    sm.abort = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    // the first tile is requested at once (nothing below touches the rows that it brings)
    pdl_wait();
    load_k(0);
    if (!fused) load_q0();
    load_v(0);
  }
  if (warp == kCtrlWarp) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&sm.tmem_base)),
                 "r"(TMEM_COLS)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  float* denbuf = reinterpret_cast<float*>(smem + off_den(z3));
  for (int idx = tid; idx < (int)ones_bytes(z3) / 16; idx += kThreads) {       // the block of ones: column 0 <- 1, the others <- 0
    const bool first = z3 ? (idx & 7) == ((idx >> 3) & 7) : (idx & 8) == 0;
    reinterpret_cast<uint4*>(smem + OFF_ONES)[idx] = make_uint4(first ? 0x3f80u : 0u, 0u, 0u, 0u);
  }
  if (GRP && tid < TILE) zs[tid] = 0.f;
  if (GRP && tstep < TILE) {                                                   // partly filled tiles: rows tstep-127 of V <- 0
    const int per_box = (TILE - tstep) * 8;                                    // 16-byte pieces per box
    for (int idx = tid; idx < 4 * per_box; idx += kThreads)
      reinterpret_cast<uint4*>(smem + vbox((idx / per_box) >> 1, (idx / per_box) & 1) + tstep * 128)[idx % per_box] = make_uint4(0u, 0u, 0u, 0u);
  }
  for (int idx = tid; idx < 4 * 1024 / 16; idx += kThreads)                    // rows 128-135 of the four K boxes <- 0
    reinterpret_cast<uint4*>(smem + OFF_K0 + (idx >> 6) * KBOX_BYTES + BOX_BYTES)[idx & 63] = make_uint4(0u, 0u, 0u, 0u);
  // The taps, for group B, and the rows before the first tile, for those who copy them: `nt` threads, t of them this one.
  auto load_taps = [&](int t, int nt) {
    for (int idx = t; idx < (LONG ? (int)long_taps(W) : W) * D; idx += nt)
      wsm[idx] = idx < W * D ? w[((size_t)h * D + (idx % D)) * W + idx / D] : 0.f;
  };
  auto load_window = [&](int t, int nt) {
    if (LONG) {                                  // [long_taps - 1][128]: zeros, then the W-1 rows of the window
      const int lead = ((int)long_taps(W) - W) * D;
      for (int idx = t; idx < ((int)long_taps(W) - 1) * D; idx += nt)
        halo0[idx] = has_in && idx >= lead ? win_in[idx - lead] : __float2bfloat16_rn(0.f);
    } else {
      for (int idx = t; idx < (W - 1) * 16; idx += nt)
        *reinterpret_cast<uint4*>(smem + off_halo(W) + halo_at(idx >> 4, idx & 15, W)) =
            has_in ? reinterpret_cast<const uint4*>(win_in)[idx] : make_uint4(0u, 0u, 0u, 0u);
    }
  };
  if constexpr (GRP) {                            // (by everybody, ahead of the barrier: the other way costs these kernels registers)
    pdl_wait();
    load_taps(tid, kThreads);
    load_window(tid, kThreads);
  }
  fence_proxy_async();
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  if (!GRP) pdl_wait();                           // everything above touched shared memory and TMEM only
  if (early) pdl_trigger();
  if (tid == kCopyWarp * 32 && nchunks > 1) {
    load_k(1);
    load_v(1);
  }
  if constexpr (!GRP) {                           // nobody else waits for these loads (group B: a barrier of its own)
    if (warp < 8) load_taps(tid, kThreadsB);
    if (LONG ? warp < 8 : warp == kHaloWarp) load_window(LONG ? tid : lane, LONG ? kThreadsB : 32);
    __syncwarp();
  }
  const uint32_t tmem = sm.tmem_base;

  // phi on rows 16 I0 ... 16 I1 - 1 of the K tile of tile m, in place, by 256 threads (ta); rows at or beyond the end of the
  // sequence become zero
  auto phi_k = [&](auto i0c, auto i1c, int m, int ta) {
    constexpr int I0 = decltype(i0c)::value, I1 = decltype(i1c)::value, NI = I1 - I0;
    if constexpr (NI > 0) {
      const int valid = min(tstep, T - m * tstep);
      const int ct = ta & 15, rg = ta >> 4;                     // chunk column 0..15, row group 0..15
      if constexpr (kRollE) {                                   // (16 rows further on the swizzle is the same)
        unsigned char* Kb = smem + ((m & 1) ? OFF_K1 : OFF_K0) + (ct >> 3) * KBOX_BYTES + swz(rg + 16 * I0, ct & 7);
        auto put = [&](int i, uint4 x) {
          *reinterpret_cast<uint4*>(Kb + i * 2048) = rg + 16 * (I0 + i) < valid ? phi8<PHI>(x) : make_uint4(0u, 0u, 0u, 0u);
        };
#pragma unroll 1
        for (int i = 0; i < NI; i += 2) {                       // two at a time, the loads first
          const uint4 x = *reinterpret_cast<const uint4*>(Kb + i * 2048), y = *reinterpret_cast<const uint4*>(Kb + min(i + 1, NI - 1) * 2048);
          put(i, x);
          if (i + 1 < NI) put(i + 1, y);
        }
      } else {
        unsigned char* Kb = smem + ((m & 1) ? OFF_K1 : OFF_K0) + (ct >> 3) * KBOX_BYTES;
        uint4 x[NI];                                              // all loads first: they do not wait for the stores
#pragma unroll
        for (int i = 0; i < NI; ++i) x[i] = *reinterpret_cast<const uint4*>(Kb + swz(rg + 16 * (I0 + i), ct & 7));
#pragma unroll
        for (int i = 0; i < NI; ++i) {
          const int j = rg + 16 * (I0 + i);
          *reinterpret_cast<uint4*>(Kb + swz(j, ct & 7)) = j < valid ? phi8<PHI>(x[i]) : make_uint4(0u, 0u, 0u, 0u);
        }
      }
    }
  };
  using K0c = std::integral_constant<int, 0>;
  using KAc = std::integral_constant<int, 8 - KB>;
  using K8c = std::integral_constant<int, 8>;

  // ---- state pass (fused): the sums of this segment, which the segments behind it start from ----
  if (fused && !writes_state) {
    if (warp == kCtrlWarp) {
      if (lane == 0)
        for (int n = 0; n < nchunks; ++n) {
          const uint32_t par = n & 1;
          // (phi(K) of tiles 0 and 1 may both be in place before this lane looks: a barrier per tile parity.  Its next phase
          // needs tile n + 2, which is loaded behind the product below.)
          if (!mbar_wait((bar0 + 8u * (B_ST_PHI0 + par)), (n >> 1) & 1, abort) || !mbar_wait((bar0 + 8u * (B_FULL_V0 + par)), (n >> 1) & 1, abort)) break;
          tc_fence_after();
          const uint32_t k_mn = desc_lo(sbase + (par ? OFF_K1 : OFF_K0), KBOX_BYTES), v_mn = desc_lo(sbase + vbox(par, 0), vstep(par));
#pragma unroll
          for (int ks = 0; ks < 8; ++ks) {     // [dS | dz] += phi(K)^T [V | 1]
            const uint64_t kd = desc64(k_mn + kstep_mnmajor(ks));
            mma_bf16(tmem + S_COL, kd, desc64(v_mn + kstep_mnmajor(ks)), z3 ? idesc(true, true, 144) : idesc(true, true, 128), n > 0 || ks > 0);
            if (!z3) mma_bf16(tmem + Z_COL, kd, desc_ext(sbase + OFF_ONES, ks), idesc(true, true, 16), n > 0 || ks > 0);
          }
          mma_commit((bar0 + 8u * (B_ST_MMA0 + par)));
        }
    } else if (warp == kCopyWarp) {
      if (lane == 0)
        for (int n = 0; n + 2 < nchunks; ++n) {
          if (!mbar_wait((bar0 + 8u * (B_ST_MMA0 + (n & 1))), (n >> 1) & 1, abort)) break;
          load_k(n + 2);
          load_v(n + 2);
        }
    } else if (warp < 16) {
      using K4c = std::integral_constant<int, 4>;
      bool ok = true;
      const int q4 = warp & 3, hf = (warp >> 2) & 1, r0 = 32 * q4 + 16 * (warp >> 3);
      const size_t at = (size_t)(r0 + (lane >> 2)) * D + 64 * hf + 2 * (lane & 3);
      const bool base = init && sg == 0;          // the first segment's sums take the caller's state in
      uint32_t x[32];
      if (base) frag_load(S + (size_t)bh * D * D + at, x);
      for (int n = 0; n < nchunks; ++n) {
        ok = ok && mbar_wait((bar0 + 8u * ((n & 1) ? B_FULL_K1 : B_FULL_K0)), (n >> 1) & 1, abort);
        ok = __all_sync(0xffffffffu, ok);
        if (ok) {
          if (warp < 8) phi_k(K0c{}, K4c{}, n, tid);
          else phi_k(K4c{}, K8c{}, n, tid - kThreadsB);
        }
        fence_proxy_async();
        mbar_arrive((bar0 + 8u * (B_ST_PHI0 + (n & 1))));
      }
      const int l = nchunks - 1;                  // (the last product; its barrier is at most one phase behind here: tile l
                                                  // was loaded only after product l - 2 had completed)
      ok = ok && mbar_wait((bar0 + 8u * (B_ST_MMA0 + (l & 1))), (l >> 1) & 1, abort);
      ok = __all_sync(0xffffffffu, ok);
      if (ok) {
        tc_fence_after();
        const size_t mine = (size_t)bh * nseg + sg;
        uint32_t v[32];
        LA_TMEM_LD_FRAG8(tmem + ((uint32_t)r0 << 16) + S_COL + 64 * hf, v);
        tmem_wait_ld();
        if (base) frag_add(v, x);
        frag_store(S_seg + mine * D * D + at, v);
        if (warp < 4) {
          const uint32_t zz = tmem_ld1(tmem + ((uint32_t)(32 * q4) << 16) + Z_COL);
          tmem_wait_ld();
          z_seg[mine * D + tid] = __uint_as_float(zz) + (base ? z[(size_t)bh * D + tid] : 0.f);
        }
      }
    }
    fence_proxy_async();                          // phi(K) in place: the buffers are loaded anew
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (tid == kCopyWarp * 32) {                  // start the main pass with fresh barriers for K and V
      for (int i : {B_FULL_K0, B_FULL_K1, B_FULL_V0, B_FULL_V1}) {
        mbar_inval(bar0 + 8u * i);
        mbar_init(bar0 + 8u * i, 1);
      }
      asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
      load_k(0);
      load_q0();
    }
  } else if (fused && tid == kCopyWarp * 32) {
    load_q0();
  }
  if (fused) {                                    // the sums are in the workspace, for every block of the chain
    cluster_arrive();
    cluster_wait();
  }

  if (has_in && warp < 16) {
    // The incoming state: fp32 into TMEM and a bf16 copy into shared memory; z: row 128 of the first K buffer (feature tid).
    // Both groups share it out, 16 rows x 64 columns per warp.
    const int q4 = warp & 3, hf = (warp >> 2) & 1, r0 = 32 * q4 + 16 * (warp >> 3);
    const size_t at = (size_t)(r0 + (lane >> 2)) * D + 64 * hf + 2 * (lane & 3);
    uint32_t v[2][16];                              // 32 columns each
#pragma unroll
    for (int hh = 0; hh < 2; ++hh) {
      auto load = [&](int j, uint32_t (&y)[16]) {
#pragma unroll
        for (int g = 0; g < 4; ++g)
#pragma unroll
          for (int i = 0; i < 2; ++i) {
            const float2 t = *reinterpret_cast<const float2*>(S_in + (size_t)j * D * D + at + i * 8 * D + 32 * hh + 8 * g);
            y[4 * g + 2 * i] = __float_as_uint(t.x);
            y[4 * g + 2 * i + 1] = __float_as_uint(t.y);
          }
      };
      auto add = [&](const uint32_t (&y)[16]) {
#pragma unroll
        for (int e = 0; e < 16; ++e) v[hh][e] = __float_as_uint(__uint_as_float(v[hh][e]) + __uint_as_float(y[e]));
      };
      load(0, v[hh]);
#pragma unroll 1
      for (int j = 1; j < nsum; j += 3) {           // the sums of the segments before this one, in order, three in flight
        uint32_t x0[16], x1[16], x2[16];
        load(j, x0);
        if (j + 1 < nsum) load(j + 1, x1);
        if (j + 2 < nsum) load(j + 2, x2);
        add(x0);
        if (j + 1 < nsum) add(x1);
        if (j + 2 < nsum) add(x2);
      }
    }
#pragma unroll
    for (int hh = 0; hh < 2; ++hh) {
      LA_TMEM_ST_FRAG4(tmem + ((uint32_t)r0 << 16) + S_COL + 64 * hf + 32 * hh, v[hh]);
#pragma unroll
      for (int g = 0; g < 4; ++g)
#pragma unroll
        for (int i = 0; i < 2; ++i)
          *reinterpret_cast<uint32_t*>(smem + OFF_S + hf * BOX_BYTES + swz(r0 + (lane >> 2) + 8 * i, 4 * hh + g) + 4 * (lane & 3)) =
              pack2(__uint_as_float(v[hh][4 * g + 2 * i]), __uint_as_float(v[hh][4 * g + 2 * i + 1]));
    }
    if (warp < 4) {                                 // z, and zeros in the other columns of its block (32 rows per warp)
      const uint32_t zaddr = tmem + ((uint32_t)(32 * q4) << 16) + Z_COL;
      const float zz = z_start(tid);
      if (GRP) zs[tid] = zz;
      else
        *reinterpret_cast<__nv_bfloat16*>(smem + OFF_K0 + (tid >> 6) * KBOX_BYTES + BOX_BYTES + (tid & 63) * 2) = __float2bfloat16_rn(zz);
      tmem_st1(zaddr, __float_as_uint(zz));
#pragma unroll
      for (int c = 1; c < 16; ++c) tmem_st1(zaddr + c, 0u);
    }
    tmem_wait_st();
    fence_proxy_async();
    tc_fence_before();
    asm volatile("bar.sync 6, 544;" ::: "memory");
    tc_fence_after();
  } else if (has_in && warp == kCopyWarp) {
    asm volatile("bar.sync 6, 544;" ::: "memory");
  }
  // (fused: V of the first tile and the second tile are requested behind the state, which would otherwise wait for them)
  if (fused && !writes_state && tid == kCopyWarp * 32) {
    load_v(0);
    if (nchunks > 1) {
      load_k(1);
      load_v(1);
    }
  }
  if (fused) cluster_arrive();                    // this block has read the caller's state (and its window)

  // S and z after tile n, which is not the last: the bf16 copy and the z row for the next tile.  256 threads (row r, 64
  // columns each): group B or group A.
  auto snapshot = [&](int n, int r, int hf, uint32_t lane_addr, bool& ok) {
    const uint32_t par = n & 1;
    unsigned char* Sb = smem + OFF_S + hf * BOX_BYTES;
    auto mbar_wait = [](uint32_t bar, uint32_t parity, volatile int* abort) {
      return la::mbar_wait<(SNAP_A ? TIGHT_A : TIGHT_B)>(bar, parity, abort);
    };
    // S_n is final after MMA_S; the old copy may be overwritten once O = phi(Q) S_prev has read it
    ok = ok && mbar_wait((bar0 + 8u * (par ? B_MMA_S1 : B_MMA_S0)), (n >> 1) & 1, abort) && mbar_wait((bar0 + 8u * (B_MMA_Q)), par, abort);
    ok = __all_sync(0xffffffffu, ok);
    if (ok) {
      tc_fence_after();
      uint32_t zbits = 0u;
      if (hf == 0) zbits = tmem_ld1(tmem + lane_addr + Z_COL);
#pragma unroll (kRoll ? 1 : 2)
      for (int qq = 0; qq < 2; ++qq) {
        uint32_t v[32];
        LA_TMEM_LD32(tmem + lane_addr + S_COL + 64 * hf + 32 * qq, v);
        tmem_wait_ld();
#pragma unroll
        for (int c = 0; c < 4; ++c) *reinterpret_cast<uint4*>(Sb + swz(r, 4 * qq + c)) = pack8(v + 8 * c);
      }
      if (hf == 0) {
        const float zz = __uint_as_float(zbits);
        if (GRP) {
          zs[r] = zz;                             // fp32, for phi(q) . z of the next tile
        } else {                                  // row 128 of the K buffer of tile n+1
          *reinterpret_cast<__nv_bfloat16*>(smem + (((n + 1) & 1) ? OFF_K1 : OFF_K0) + (r >> 6) * KBOX_BYTES + BOX_BYTES +
                                            (r & 63) * 2) = __float2bfloat16_rn(zz);
        }
      }
    }
    fence_proxy_async();
    tc_fence_before();
    mbar_arrive((bar0 + 8u * (B_SB)));
  };

  if (warp >= 16) {
  if (TRADE) regs_down<64>();
  auto mbar_wait = [](uint32_t bar, uint32_t parity, volatile int* abort) { return la::mbar_wait<TIGHT_C>(bar, parity, abort); };
  if (warp == kCtrlWarp) {
    // =============================== MMA issue, the Q and K loads (one lane) ===============================
    if (lane == 0) {
      bool ok = true;
      for (int n = 0; n < nchunks; ++n) {
        const uint32_t par = n & 1;
        const uint32_t vbuf = sbase + vbox(par, 0);
        const uint32_t kbuf = sbase + (par ? OFF_K1 : OFF_K0);
        const bool has_state = has_in || n > 0;
        // low descriptor words of step 0: K read along its rows (K-major), K, V and the S copy down their rows
        const uint32_t k_km = desc_lo(kbuf, 16u);
        const uint32_t k_mn = desc_lo(kbuf, KBOX_BYTES), v_mn = desc_lo(vbuf, vstep(par)), s_mn = desc_lo(sbase + OFF_S, BOX_BYTES);
        if (GRP) {
          // scores of the raw q and k, both operands from shared memory as TMA delivered them; group A applies phi
          // only once this product is complete
          ok = mbar_wait((bar0 + 8u * (B_FULL_Q)), par, abort) &&
               mbar_wait((bar0 + 8u * (par ? B_FULL_K1 : B_FULL_K0)), (n >> 1) & 1, abort);
          if (!ok) break;
          const uint32_t q_km = desc_lo(sbase + OFF_Q, 16u);
#pragma unroll
          for (int ks = 0; ks < 8; ++ks)
            mma_bf16(tmem + P_COL, desc64(q_km + kstep_kmajor(ks)), desc64(k_km + kstep_kmajor(ks, KBOX_BYTES)),
                     idesc(false, false, 128), ks > 0);
          mma_commit((bar0 + 8u * (B_MMA_P)));
        }
        // phi(Q) of tile n is in TMEM, phi(K) in place; the copy of S and z before tile n are complete (after n + 1 arrivals:
        // from here on the update may change S)
        ok = mbar_wait((bar0 + 8u * (B_PHI)), par, abort) && mbar_wait((bar0 + 8u * (B_SB)), par, abort);
        if (!ok) break;
        tc_fence_after();
        // The Q buffer has been read by then (phi(Q) lives in TMEM): its reload, which sets the pace, goes out first.
        if (n + 1 < nchunks) {
          mbar_expect_tx((bar0 + 8u * (B_FULL_Q)), tile_tx);
          tma_load(sbase + OFF_Q, &mq, 0, y0 + (n + 1) * tstep, bh, (bar0 + 8u * (B_FULL_Q)));
          tma_load(sbase + OFF_Q + BOX_BYTES, &mq, 64, y0 + (n + 1) * tstep, bh, (bar0 + 8u * (B_FULL_Q)));
        }
        if (MULTI) {                       // the scores of rows gsz (c + 1) ... 127 against the tokens of group c of this tile
          if (use_glob)
            for (int c = 0; c + 1 < TILE / gsz; ++c)
#pragma unroll
              for (int ks = 0; ks < 8; ++ks)
                mma_bf16_ts_below(tmem + P_COL + gsz * c, tmem + FQ_COL + 8 * ks,
                                  desc64(k_km + (((uint32_t)(gsz * c) * 128u) >> 4) + kstep_kmajor(ks, KBOX_BYTES)),
                                  idesc(false, false, (uint32_t)gsz), ks > 0, gsz * (c + 1));
          mma_commit((bar0 + 8u * (B_MMA_L)));
        }
        if (!GRP) {
#pragma unroll
          for (int ks = 0; ks < 8; ++ks)   // [P | phi(q).z_prev] = phi(Q) [phi(K); z_prev]^T; 16 channels of phi(Q) = 8 columns
            mma_bf16_ts(tmem + P_COL, tmem + FQ_COL + 8 * ks, desc64(k_km + kstep_kmajor(ks, KBOX_BYTES)),
                        idesc(false, false, 144), ks > 0);
          mma_commit((bar0 + 8u * (B_MMA_P)));
        }
        // The state update needs nothing from the previous tile's epilogue: it fills the time until that epilogue
        // has read the accumulator.
        ok = mbar_wait((bar0 + 8u * (B_FULL_V0 + par)), (n >> 1) & 1, abort);
        if (!ok) break;
#pragma unroll
        for (int ks = 0; ks < 8; ++ks) {     // [S | z] += phi(K)^T [V | 1]
          const uint64_t kd = desc64(k_mn + kstep_mnmajor(ks));
          mma_bf16(tmem + S_COL, kd, desc64(v_mn + kstep_mnmajor(ks)), z3 ? idesc(true, true, 144) : idesc(true, true, 128),
                   has_state || ks > 0);
          if (!z3) mma_bf16(tmem + Z_COL, kd, desc_ext(sbase + OFF_ONES, ks), idesc(true, true, 16), has_state || ks > 0);
        }
        mma_commit((bar0 + 8u * (par ? B_MMA_S1 : B_MMA_S0)));
        // the accumulator is free once the epilogue of tile n-1 has read it
        if (n >= 1) ok = mbar_wait((bar0 + 8u * (B_EPI0 + (par ^ 1))), ((n - 1) >> 1) & 1, abort);
        if (!ok) break;
        tc_fence_after();
        if (has_state && (!GRP || use_glob)) {
#pragma unroll
          for (int ks = 0; ks < 8; ++ks)     // O = phi(Q) S_prev
            mma_bf16_ts(tmem + O_COL, tmem + FQ_COL + 8 * ks, desc64(s_mn + kstep_mnmajor(ks)), idesc(false, true, 128), ks > 0);
        }
        mma_commit((bar0 + 8u * (B_MMA_Q)));
        ok = mbar_wait((bar0 + 8u * (B_PDONE)), par, abort);               // masked P of tile n is in TMEM
        if (!ok) break;
        tc_fence_after();
        if (MULTI) {
          // A group's tokens meet its own rows and those below: the rows above are masked off, and not met with zeros, which
          // would give them a NaN where v of a later group is not finite.  16 tokens of every row of P = 8 columns; then the
          // remainders of the linear scores, for the rows below the group.
          // (The masks as constants, a copy of the code per group size: as numbers of the run they cost 2 % of a pass.)
          const int valid = min(TILE, T - n * TILE);
          auto products = [&](auto gc) {
            constexpr int G = decltype(gc)::value;
#pragma unroll
            for (int ks = 0; ks < 8; ++ks)
              if (16 * ks < valid)
                mma_bf16_ts_below(tmem + O_COL, tmem + P_COL + 16 * ks, desc64(v_mn + kstep_mnmajor(ks)), idesc(false, true, 128),
                                  (has_state && use_glob) || ks > 0, 16 * ks / G * G);
#pragma unroll
            for (int ks = 0; 16 * ks < TILE - G; ++ks)
              if (use_glob && (16 * ks / G + 1) * G < valid)
                mma_bf16_ts_below(tmem + O_COL, tmem + P_COL + 16 * ks + 8, desc64(v_mn + kstep_mnmajor(ks)),
                                  idesc(false, true, 128), true, (16 * ks / G + 1) * G);
          };
          if (gsz == 64) products(std::integral_constant<int, 64>{});
          else products(std::integral_constant<int, 32>{});
        } else {
#pragma unroll
          for (int ks = 0; ks < 8; ++ks)     // O += (P o M) V; 16 tokens of every row of P = 8 columns
            mma_bf16_ts(tmem + O_COL, tmem + P_COL + (ks < 4 ? 8 * ks : 64 + 8 * (ks - 4)), desc64(v_mn + kstep_mnmajor(ks)),
                        idesc(false, true, 128), (has_state && (!GRP || use_glob)) || ks > 0);
        }
        mma_commit((bar0 + 8u * (B_MMA_O0 + par)));
        // P of the next tile overwrites the columns that the last product of this tile reads
        ok = mbar_wait((bar0 + 8u * (B_MMA_O0 + par)), (n >> 1) & 1, abort);
        if (!ok) break;
      }
    }
  } else if (warp == kCopyWarp) {
    // =============================== V reloads and output stores (lane 0), K reloads (lane 1) ===============================
    // A lane of its own, so that waiting for a store to have read its buffer never holds up the issue of products.
    if (lane == 0) {
      bool ok = true;
      for (int n = 0; n < nchunks; ++n) {
        const uint32_t par = n & 1;
        // the outputs of tile n are staged in its V buffer: store them; once they have been read the buffer takes
        // tile n+2
        ok = mbar_wait((bar0 + 8u * (B_STAGED0 + par)), (n >> 1) & 1, abort);
        if (!ok) break;
        const uint32_t vb = sbase + vbox(par, 0), vb1 = sbase + vbox(par, 1);
        if (LONG) {
          // the outputs wait in the token rows of this tile's K buffer; every tap has been taken from its V buffer
          const uint32_t kb = sbase + (par ? OFF_K1 : OFF_K0);
          tma_store(&mo, 0, y0 + n * tstep, bh, kb);
          tma_store(&mo, 64, y0 + n * tstep, bh, kb + KBOX_BYTES);
          tma_commit();
          if (n + 2 < nchunks) {
            load_v(n + 2);
            tma_wait_read();
            load_k(n + 2);
          }
          continue;
        }
        tma_store(&mo, 0, y0 + n * tstep, bh, vb);               // rows past the end of the sequence are clipped
        tma_store(&mo, 64, y0 + n * tstep, bh, vb1);
        tma_commit();
        if (n + 2 < nchunks) {
          tma_wait_read();
          load_v(n + 2);
        }
      }
      tma_wait_all();                             // every store is complete before the CTA exits
    } else if (lane == 1 && !LONG) {
      // A lane of its own for the K reloads (short-window mode): the K buffer of tile n is free the moment its state
      // update completes, and phi(K) of tile n+2 is wanted early -- neither the issuing lane nor the store lane
      // should have to stand by for that moment.
      for (int n = 0; n + 2 < nchunks; ++n) {
        const uint32_t par = n & 1;
        if (!mbar_wait((bar0 + 8u * (par ? B_MMA_S1 : B_MMA_S0)), (n >> 1) & 1, abort)) break;
        load_k(n + 2);
      }
    }
  } else if (warp == kHaloWarp) {
    // =============================== the rows of v before every 32 rows (short windows) ===============================
    // The epilogue overwrites V with the outputs 32 rows at a time, without waiting for its other warps: what the taps of
    // the next 32 rows (or of the next tile) reach back to is copied aside first.
    if constexpr (WT > 1) {
      bool ok = true;
      for (int n = 0; n < nchunks; ++n) {
        const uint32_t par = n & 1;
        const int valid = min(tstep, T - n * tstep);
        ok = ok && mbar_wait((bar0 + 8u * (B_FULL_V0 + par)), (n >> 1) & 1, abort);
        ok = __all_sync(0xffffffffu, ok);
        if (ok) {
          unsigned char* hb = smem + off_halo(WT);
          uint4 x[2 * (WT - 1)];
#pragma unroll
          for (int m = 0; m < 2 * (WT - 1); ++m) {          // piece lane & 15 of rows 2 m, 2 m + 1 of the 4 (W - 1)
            const int j = 2 * m + (lane >> 4), blk = j / (WT - 1), i = j % (WT - 1);
            const int row = (blk < 3 ? 32 * (blk + 1) : valid) - (WT - 1) + i;
            x[m] = row >= 0 ? *reinterpret_cast<const uint4*>(smem + vbox(par, (lane & 15) >> 3) + swz(row, lane & 7))
                            : *reinterpret_cast<const uint4*>(hb + (n % 3) * halo_bytes(WT) + halo_at(row + WT - 1, lane & 15, WT));
          }
#pragma unroll
          for (int m = 0; m < 2 * (WT - 1); ++m) {
            const int j = 2 * m + (lane >> 4), blk = j / (WT - 1), i = j % (WT - 1);
            const int buf = blk < 3 ? 3 + 3 * (int)par + blk : (n + 1) % 3;
            *reinterpret_cast<uint4*>(hb + buf * halo_bytes(WT) + halo_at(i, lane & 15, WT)) = x[m];
          }
          __syncwarp();                                     // (a short last tile reads rows that other lanes wrote here)
        }
        mbar_arrive((bar0 + 8u * (B_HALO0 + par)));
      }
    }
  }
  } else if (warp >= 8) {
    // =============================== group A: phi, P, [S|z] snapshot (256 threads) ===============================
    auto mbar_wait = [](uint32_t bar, uint32_t parity, volatile int* abort) { return la::mbar_wait<TIGHT_A>(bar, parity, abort); };
    if constexpr (TRADE) {
      if constexpr (kRegsA > 96) regs_up<kRegsA>();
      if constexpr (kRegsA < 96) regs_down<kRegsA>();
    }
    const int ta = tid - kThreadsB;               // 0..255
    const int wa = warp - 8;                      // 0..7
    const int r = 32 * (wa & 3) + lane;           // tile row = TMEM lane
    const int hf = wa >> 2;                       // column half
    const uint32_t lane_addr = (uint32_t)(32 * (wa & 3)) << 16;
    unsigned char* Qb = smem + OFF_Q + hf * BOX_BYTES;
    bool ok = true;

    if (SNAP_A) mbar_arrive((bar0 + 8u * (B_SB)));           // phase 0: the state before tile 0 is in place

    if (!GRP) {
      ok = mbar_wait((bar0 + 8u * (B_FULL_K0)), 0, abort);
      ok = __all_sync(0xffffffffu, ok);
      if (ok) phi_k(K0c{}, KAc{}, 0, ta);
    }

    for (int n = 0; n < nchunks; ++n) {
      const uint32_t par = n & 1;
      const bool last = n + 1 == nchunks;

      // ---- phi on Q in place (phi on K of this tile was done one iteration earlier) ----
      ok = ok && mbar_wait((bar0 + 8u * (B_FULL_Q)), par, abort);
      if (GRP) ok = ok && mbar_wait((bar0 + 8u * (B_SB)), par, abort);       // z before tile n is in place
      ok = __all_sync(0xffffffffu, ok);
      if (GRP) sync_group_a();                    // every thread is done with the halves of the last tile (dgh, mlh)
      // phi(q) of row r, this thread's 64 channels: 32 packed pairs = 32 TMEM columns of lane r.
      uint32_t fq[kRoll ? 16 : 32];
      float dg = 0.f;
      auto phi_q = [&](int c0) {                  // pieces c0 ... of the row
#pragma unroll
        for (int cc = 0; cc < (kRoll ? 4 : 8); ++cc) {
          const uint4 f = phi8<PHI>(*reinterpret_cast<const uint4*>(Qb + swz(r, c0 + cc)));
          fq[4 * cc] = f.x; fq[4 * cc + 1] = f.y; fq[4 * cc + 2] = f.z; fq[4 * cc + 3] = f.w;
        }
      };
      if (ok && !kRoll) phi_q(0);
      if (!SNAP_A) {                              // the products of tile n-1 that read these columns are complete
        if (n > 0) ok = ok && mbar_wait((bar0 + 8u * (B_MMA_Q)), par ^ 1, abort);
        ok = __all_sync(0xffffffffu, ok);
        tc_fence_after();
      }
      if (ok) {
        if constexpr (!kRoll) {
          LA_TMEM_ST32(tmem + lane_addr + FQ_COL + 32 * hf, fq);
        } else {
#pragma unroll 1
          for (int qq = 0; qq < 2; ++qq) {
            phi_q(4 * qq);
            LA_TMEM_ST16(tmem + lane_addr + FQ_COL + 32 * hf + 16 * qq, fq);
          }
        }
        if constexpr (GRP) {                      // this half of phi(q) . z_prev, z in fp32
#pragma unroll
          for (int e = 0; e < 32; e += 2) {
            const float4 z4 = *reinterpret_cast<const float4*>(zs + 64 * hf + 2 * e);
            dg = fmaf(lo_f(fq[e]), z4.x, fmaf(hi_f(fq[e]), z4.y, fmaf(lo_f(fq[e + 1]), z4.z, fmaf(hi_f(fq[e + 1]), z4.w, dg))));
          }
          if (!MULTI) dgh[hf * D + r] = dg;
        }
        tmem_wait_st();
      }
      if (GRP) {
        // phi on K of this tile, in place: the score product runs on the raw q and k, so K may be touched only once
        // that product is complete (phi(Q) above reads the Q buffer and writes TMEM: it ran beside the product)
        ok = ok && mbar_wait((bar0 + 8u * (par ? B_FULL_K1 : B_FULL_K0)), (n >> 1) & 1, abort) &&
             mbar_wait((bar0 + 8u * (B_MMA_P)), par, abort);
        ok = __all_sync(0xffffffffu, ok);
        if (ok) phi_k(K0c{}, K8c{}, n, ta);
      }
      fence_proxy_async();                        // (phi(K) of this tile, written one iteration earlier)
      tc_fence_before();
      mbar_arrive((bar0 + 8u * (B_PHI)));
      float dpart = 0.f;                          // this half of the row sum of the masked P

      // ---- phi on K of the next tile, while the tensor cores form the scores of this one.  (Not with the long-window
      //      epilogue: there the K buffer comes back late, after the outputs staged in it have left, and waiting for
      //      it here would hold up the mask; see below.) ----
      if (!GRP && !LONG && !last) {
        ok = ok && mbar_wait((bar0 + 8u * (((n + 1) & 1) ? B_FULL_K1 : B_FULL_K0)), ((n + 1) >> 1) & 1, abort);
        ok = __all_sync(0xffffffffu, ok);
        if (ok) phi_k(K0c{}, KAc{}, n + 1, ta);
      }

      // ---- P: causal mask, packed bf16 -> TMEM ----
      if (!GRP) ok = ok && mbar_wait((bar0 + 8u * (B_MMA_P)), par, abort);
      ok = __all_sync(0xffffffffu, ok);
      if (!GRP && ok) {
        tc_fence_after();
#pragma unroll (kRoll ? 1 : 2)
        for (int qq = 0; qq < 2; ++qq) {
          const int col0 = 64 * hf + 32 * qq;
          uint32_t v[32], pk[16];
          float ps0 = 0.f, ps1 = 0.f;
          if (col0 <= 32 * (wa & 3) + 31) {                     // warp-uniform: some row of this warp reaches col0
            LA_TMEM_LD32(tmem + P_COL + lane_addr + col0, v);
            tmem_wait_ld();
#pragma unroll
            for (int e = 0; e < 16; ++e) {
              const float p0 = col0 + 2 * e <= r ? __uint_as_float(v[2 * e]) : 0.f;
              const float p1 = col0 + 2 * e + 1 <= r ? __uint_as_float(v[2 * e + 1]) : 0.f;
              pk[e] = pack2(p0, p1);
              ps0 += p0;
              ps1 += p1;
            }
            dpart += ps0 + ps1;
          } else {
#pragma unroll
            for (int e = 0; e < 16; ++e) pk[e] = 0u;
          }
          LA_TMEM_ST16(tmem + P_COL + lane_addr + 64 * hf + 16 * qq, pk);
        }
        if (hf == 1) {                            // phi(q) . z_prev, delivered by the score product as column 128
          dpart += __uint_as_float(tmem_ld1(tmem + lane_addr + QZ_COL));
          tmem_wait_ld();
        }
        // (slot n & 1 was last read by the epilogue of tile n-2, before the arrival that released the accumulator to
        // tile n-1, whose products were complete before P of this tile was issued)
        denbuf[(par * 2 + hf) * D + r] = dpart;
        tmem_wait_st();
      }
      if constexpr (MULTI) {
        // ---- P: causal softmax inside the row's group (the two threads of a row take half of its columns each), the
        // linear scores against the earlier groups of the tile (nothing behind the group: no product reads it).
        const float c2 = sm_scale * 1.4426950408889634f;       // scores -> exponents of two
        const int b0 = 32 * (wa & 3) / gsz * gsz, hw = gsz >> 1, d0 = b0 + hw * hf, l0 = (b0 >> 1) * hf;   // warp-uniform
        float m_run = -INFINITY, l_run = 0.f;
        const uint32_t pbase = tmem + P_COL + lane_addr;
        uint32_t v[32];
        if (ok) {
          tc_fence_after();
          if (hw == 32) LA_TMEM_LD32(tmem + P_COL + lane_addr + d0, v);
          else LA_TMEM_LD16(tmem + P_COL + lane_addr + d0, v);
          tmem_wait_ld();
#pragma unroll
          for (int e = 0; e < 32; ++e) {
            v[e] = __float_as_uint((e < 16 || hw == 32) && d0 + e <= r ? __uint_as_float(v[e]) * c2 : -INFINITY);
            m_run = fmaxf(m_run, __uint_as_float(v[e]));
          }
          if (m_run > -INFINITY) {
#pragma unroll
            for (int e = 0; e < 32; ++e) l_run += ex2(__uint_as_float(v[e]) - m_run);
          }
        }
        if (use_glob && b0 > 0) {
          ok = ok && mbar_wait((bar0 + 8u * (B_MMA_L)), par, abort);
          ok = __all_sync(0xffffffffu, ok);
        }
#pragma unroll
        for (int c = 0; c < 3; ++c)                             // 16 of this thread's b0 / 2 linear scores at a time
          if (32 * c < b0 && ok) {
            uint32_t x[16], hi[8], lo[8];
#pragma unroll
            for (int e = 0; e < 16; ++e) x[e] = 0u;
            if (use_glob) {
              tc_fence_after();
              LA_TMEM_LD16(pbase + l0 + 16 * c, x);
              tmem_wait_ld();
            }
#pragma unroll
            for (int e = 0; e < 8; ++e) {
              const float x0 = __uint_as_float(x[2 * e]), x1 = __uint_as_float(x[2 * e + 1]);
              hi[e] = pack2(x0, x1);
              lo[e] = pack2(x0 - lo_f(hi[e]), x1 - hi_f(hi[e]));
              dg += x0 + x1;
            }
            tmem_st8(pbase + l0 + 16 * c, hi);
            if (use_glob) tmem_st8(pbase + l0 + 16 * c + 8, lo);
          }
        mlh[hf * D + r] = make_float2(m_run, l_run);
        dgh[hf * D + r] = dg;
        tc_fence_before();
        sync_group_a();
        const float2 oth = mlh[(hf ^ 1) * D + r];
        const float m = fmaxf(m_run, oth.x);                    // finite: the row's own column lies in one of the halves
        const float l = l_run * ex2(m_run - m) + oth.y * ex2(oth.x - m);
        const float den = dgh[r] + dgh[D + r] + eps;
        const bool has_g = use_glob && (has_in || n > 0 || b0 > 0) && den != 0.f;
        const float rs = has_g ? den / alpha : 1.f, f = rs / l;
        if (ok) {
          tc_fence_after();
          uint32_t pk[16];
#pragma unroll
          for (int e = 0; e < 16; ++e)
            pk[e] = pack2(ex2(__uint_as_float(v[2 * e]) - m) * f, ex2(__uint_as_float(v[2 * e + 1]) - m) * f);
          tmem_st8(pbase + d0, pk);
          if (hw == 32) tmem_st8(pbase + d0 + 16, pk + 8);
          denbuf[(par * 2 + hf) * D + r] = hf == 0 ? rs : 0.f;
          tmem_wait_st();
        }
      } else if (GRP) {
        // ---- P: causal softmax along the rows.  A row's 128 columns belong to two threads (halves): each takes the
        // running maximum and sum of its half, the halves meet through shared memory, and a second pass writes
        // exp(s - max) / sum back as bf16 -- times (phi(q) . z_prev + eps) / alpha where the global branch is alive, so
        // that the epilogue's one row factor alpha / (phi(q) . z_prev + eps) finishes both branches.
        const float c2 = sm_scale * 1.4426950408889634f;       // scores -> exponents of two
        float m_run = -INFINITY, l_run = 0.f;
        if (ok) {
          tc_fence_after();
#pragma unroll
          for (int qq = 0; qq < 2; ++qq) {
            const int col0 = 64 * hf + 32 * qq;
            if (col0 <= 32 * (wa & 3) + 31) {                   // warp-uniform: some row of this warp reaches col0
              uint32_t v[32];
              LA_TMEM_LD32(tmem + P_COL + lane_addr + col0, v);
              tmem_wait_ld();
              float bm = -INFINITY;
#pragma unroll
              for (int e = 0; e < 32; ++e)
                if (col0 + e <= r) bm = fmaxf(bm, __uint_as_float(v[e]) * c2);
              if (bm > -INFINITY) {
                const float mn = fmaxf(m_run, bm);
                float acc = 0.f;
#pragma unroll
                for (int e = 0; e < 32; ++e)
                  if (col0 + e <= r) acc += ex2(__uint_as_float(v[e]) * c2 - mn);
                l_run = l_run * ex2(m_run - mn) + acc;
                m_run = mn;
              }
            }
          }
        }
        mlh[hf * D + r] = make_float2(m_run, l_run);
        sync_group_a();
        const float2 oth = mlh[(hf ^ 1) * D + r];
        const float m = fmaxf(m_run, oth.x);                    // finite: the row's own column lies in one of the halves
        const float l = l_run * ex2(m_run - m) + oth.y * ex2(oth.x - m);
        const float den = dgh[r] + dgh[D + r] + eps;
        const bool has_g = use_glob && (has_in || n > 0) && den != 0.f;
        const float rs = has_g ? den / alpha : 1.f;
        const float f = rs / l;
        if (ok) {
#pragma unroll
          for (int qq = 0; qq < 2; ++qq) {
            const int col0 = 64 * hf + 32 * qq;
            uint32_t pk[16];
            if (col0 <= 32 * (wa & 3) + 31) {
              uint32_t v[32];
              LA_TMEM_LD32(tmem + P_COL + lane_addr + col0, v);
              tmem_wait_ld();
#pragma unroll
              for (int e = 0; e < 16; ++e) {
                const float p0 = col0 + 2 * e <= r ? ex2(__uint_as_float(v[2 * e]) * c2 - m) * f : 0.f;
                const float p1 = col0 + 2 * e + 1 <= r ? ex2(__uint_as_float(v[2 * e + 1]) * c2 - m) * f : 0.f;
                pk[e] = pack2(p0, p1);
              }
            } else {
#pragma unroll
              for (int e = 0; e < 16; ++e) pk[e] = 0u;
            }
            LA_TMEM_ST16(tmem + P_COL + lane_addr + 64 * hf + 16 * qq, pk);
          }
          // the epilogue's row factor is 1 / (the two halves + its eps): the factor here, nothing else
          denbuf[(par * 2 + hf) * D + r] = hf == 0 ? rs : 0.f;
          tmem_wait_st();
        }
      }
      tc_fence_before();
      mbar_arrive((bar0 + 8u * (B_PDONE)));

      if (!GRP && LONG && !last) {                // long-window epilogue: phi on K of the next tile after the mask
        ok = ok && mbar_wait((bar0 + 8u * (((n + 1) & 1) ? B_FULL_K1 : B_FULL_K0)), ((n + 1) >> 1) & 1, abort);
        ok = __all_sync(0xffffffffu, ok);
        if (ok) phi_k(K0c{}, KAc{}, n + 1, ta);
      }

      if (SNAP_A && !last) snapshot(n, r, hf, lane_addr, ok);
    }

    // ---- the final state to global memory (this group has nothing else to do after the last tile) ----
    {
      const int n = nchunks - 1;
      ok = ok && mbar_wait((bar0 + 8u * ((n & 1) ? B_MMA_S1 : B_MMA_S0)), (n >> 1) & 1, abort);
      ok = __all_sync(0xffffffffu, ok);
      if (fused) cluster_wait();                  // every block of the chain has read the caller's state
      if (ok && writes_state) {
        tc_fence_after();
#pragma unroll
        for (int i = 0; i < 2; ++i) {             // rows 16 i ... 16 i + 15 of this warp's 32
          uint32_t v[32];
          LA_TMEM_LD_FRAG8(tmem + lane_addr + ((uint32_t)(16 * i) << 16) + S_COL + 64 * hf, v);
          tmem_wait_ld();
          frag_store(S + (size_t)bh * D * D + (size_t)((r & ~31) + 16 * i + (lane >> 2)) * D + 64 * hf + 2 * (lane & 3), v);
        }
        if (hf == 0) {
          const uint32_t zbits = tmem_ld1(tmem + lane_addr + Z_COL);
          tmem_wait_ld();
          z[(size_t)bh * D + r] = __uint_as_float(zbits);
        }
      }
    }
  } else {
    // =============================== group B: epilogue (256 threads) ===============================
    auto mbar_wait = [](uint32_t bar, uint32_t parity, volatile int* abort) { return la::mbar_wait<TIGHT_B>(bar, parity, abort); };
    if (TRADE && kRegsB > 96) regs_up<kRegsB>();
    if (!GRP) sync_group_b();                     // the taps (long windows: and the rows before the first tile) are in place
    const int r = 32 * (warp & 3) + lane;         // tile row = TMEM lane
    const int hf = warp >> 2;                     // column half
    const uint32_t lane_addr = (uint32_t)(32 * (warp & 3)) << 16;
    bool ok = true;
    if constexpr (LONG) {
      // Two phases per tile.  (1) Row by row, as the accumulator's lanes dictate: the attention term O / den goes,
      // rounded to bf16, into the token rows of this tile's K buffer, which every product has finished with (its
      // reload for tile n + 2 waits, in this mode, until the outputs have left).  (2) Channel pair by channel pair:
      // thread (cp, jq) owns channels 2 cp, 2 cp + 1 and rows 32 jq ... 32 jq + 31, forms the tap sums of 16 rows at a
      // time in registers (every row of v it needs is read once per group of 8 taps, and the taps of a group sit in
      // registers), adds the attention term and writes the output over it.  The shared-memory traffic of a tile no
      // longer grows with rows x taps x 16 bytes, and the V buffer is never written.
      const int cp = tid & 63, jq = tid >> 6;
      const int cc = (cp & 31) >> 2;                                         // 16-byte piece of the pair in its box row
      const uint32_t colv = (uint32_t)(cp & 3) * 4u + (uint32_t)jq * 4096u;
      const uint32_t colk = (uint32_t)(cp >> 5) * KBOX_BYTES + (uint32_t)(cp & 3) * 4u + (uint32_t)jq * 4096u;
      const int lead = (int)long_taps(W) - W;                                // rows of zeros at the head of the halo
      const uint32_t hcol = sbase + off_halo_long(W, GRP) + 4u * cp;
      const uint32_t hend = hcol + (long_taps(W) - 1) * (D * 2);
      const uint32_t wcol = sbase + off_w(z3) + 8u * cp;
      const int ngroups = ONE8 ? 1 : (W + 7) >> 3;
      for (int n = 0; n < nchunks; ++n) {
        const uint32_t par = n & 1;
        if (!early && n + 1 == nchunks) pdl_trigger();
        const int valid = min(tstep, T - n * tstep);
        const uint32_t vthr = sbase + vbox(par, cp >> 5) + colv;       // this thread's column at its first row
        unsigned char* stage = smem + (par ? OFF_K1 : OFF_K0);
        ok = ok && mbar_wait((bar0 + 8u * (B_MMA_O0 + par)), (n >> 1) & 1, abort);   // also: every product that reads K or V is done
        ok = __all_sync(0xffffffffu, ok);
        uint32_t v[32];
        float rden = 0.f;
        if (ok) {
          tc_fence_after();
          LA_TMEM_LD32(tmem + lane_addr + O_COL + 64 * hf, v);
          const float den = denbuf[(par * 2) * D + r] + denbuf[(par * 2 + 1) * D + r];
          rden = 1.f / (den + (GRP ? 0.f : eps));
        }
        unsigned char* Lb = stage + hf * KBOX_BYTES;
#pragma unroll
        for (int qq = 0; qq < 2; ++qq) {
          if (ok) {
            tmem_wait_ld();
            uint4 la[4];
#pragma unroll
            for (int c = 0; c < 4; ++c)
              la[c] = make_uint4(pack2(__uint_as_float(v[8 * c]) * rden, __uint_as_float(v[8 * c + 1]) * rden),
                                 pack2(__uint_as_float(v[8 * c + 2]) * rden, __uint_as_float(v[8 * c + 3]) * rden),
                                 pack2(__uint_as_float(v[8 * c + 4]) * rden, __uint_as_float(v[8 * c + 5]) * rden),
                                 pack2(__uint_as_float(v[8 * c + 6]) * rden, __uint_as_float(v[8 * c + 7]) * rden));
            if (qq == 0) LA_TMEM_LD32(tmem + lane_addr + O_COL + 64 * hf + 32, v);
#pragma unroll
            for (int c = 0; c < 4; ++c) *reinterpret_cast<uint4*>(Lb + swz(r, 4 * qq + c)) = la[c];
          }
        }
        tc_fence_before();
        mbar_arrive((bar0 + 8u * (B_EPI0 + par)));           // this accumulator has been read
        ok = ok && mbar_wait((bar0 + 8u * (B_FULL_V0 + par)), (n >> 1) & 1, abort);
        ok = __all_sync(0xffffffffu, ok);
        sync_group_b();                                      // the attention term of every row is in place
        if (ok) {
          uint32_t pv[8];
#pragma unroll
          for (int k = 0; k < 8; ++k) pv[k] = vthr + ((cc ^ k) << 4);
          const uint32_t sthr = sbase + (par ? OFF_K1 : OFF_K0) + colk;
          const int mine = valid - 32 * jq;                  // rows of this thread that hold tokens
          if constexpr (ONE8 || GRP) {
#pragma unroll 1
            for (int blk = 0; blk < 4 && 8 * blk < mine; ++blk) conv_rows8(blk, jq == 0, wcol, pv, sthr, cc, hend, ngroups);
          } else {
#pragma unroll 1
            for (int blk = 0; blk < 2 && 16 * blk < mine; ++blk) conv_rows(blk, jq == 0, wcol, pv, sthr, cc, hend, ngroups);
          }
          if (jq == 0) {
            // The rows before the next tile: the last W-1 of (halo ++ valid rows of v), in place.  This thread is the
            // only one that reads or writes this column of the halo (the rows of the other threads start at 32, and
            // no window reaches back further than 31 rows).
            // (Eight rows at a time: row by row, every load waited for, it took 3 K cycles of a tile at 32 taps.)
            for (int i0 = 0; i0 < W - 1; i0 += 8) {
              uint32_t x[8];
#pragma unroll
              for (int i = 0; i < 8; ++i) {
                const int src = min(valid - (W - 1) + i0 + i, valid - 1);
                x[i] = lds32(src >= 0 ? vthr + src * 128 + ((cc ^ (src & 7)) << 4) : hend + src * (D * 2));
              }
#pragma unroll
              for (int i = 0; i < 8; ++i)
                if (i0 + i < W - 1) sts32(hcol + (lead + i0 + i) * (D * 2), x[i]);
            }
          }
        }
        fence_proxy_async();
        mbar_arrive((bar0 + 8u * (B_STAGED0 + par)));
      }
    } else
    {
    // 32 rows x 64 channels per warp, as 8 x 8 fragments: a lane holds two channels of rows l >> 2, + 8, + 16, + 24 per
    // fragment column, so that one 8-byte load of a tap serves eight multiply-adds (with a row per lane every tap was
    // loaded for two).  ldmatrix brings v of row r - t for all rows at once; the outputs take the place of the V rows,
    // which no other warp reads (the halo buffers hold what reaches across), so that no barrier is needed.
    constexpr int WN = WT > 0 ? WT : 1;
    const int q4 = warp & 3;
    const uint32_t waddr = sbase + off_w(true) + 4u * (64 * hf + 2 * (lane & 3));
    if (KB > 0) {                                 // this group's share of the first K tile
      ok = mbar_wait((bar0 + 8u * (B_FULL_K0)), 0, abort);
      ok = __all_sync(0xffffffffu, ok);
      if (ok) phi_k(KAc{}, K8c{}, 0, tid);
      fence_proxy_async();
    }
    if (!SNAP_A) mbar_arrive((bar0 + 8u * (B_SB)));  // phase 0: the state before tile 0 is in place
    for (int n = 0; n < nchunks; ++n) {
      const uint32_t par = n & 1;
      const int valid = min(tstep, T - n * tstep);
      if (!early && n + 1 == nchunks) pdl_trigger();
      if (KB > 0 && n + 1 < nchunks) {            // (announced, like the state, by the arrival in snapshot)
        ok = ok && mbar_wait((bar0 + 8u * (((n + 1) & 1) ? B_FULL_K1 : B_FULL_K0)), ((n + 1) >> 1) & 1, abort);
        ok = __all_sync(0xffffffffu, ok);
        if (ok) phi_k(KAc{}, K8c{}, n + 1, tid);
      }
      if (!SNAP_A && n + 1 < nchunks) snapshot(n, r, hf, lane_addr, ok);
      uint32_t vrow[WN];                          // row lane - t of the warp's 32: this lane's address for ldmatrix, chunk 0
      {
        const uint32_t vb = sbase + vbox(par, hf) + 4096u * q4;
        const uint32_t he = sbase + off_halo(WN) + (q4 == 0 ? n % 3 : 2 + 3 * par + q4) * halo_bytes(WN) + (hf + 1) * (WN - 1) * 128u;
#pragma unroll
        for (int t = 0; t < WN; ++t) vrow[t] = (lane >= t ? vb : he) + (uint32_t)((lane - t) * 128) + (uint32_t)(((lane - t) & 7) << 4);
      }
      ok = ok && mbar_wait((bar0 + 8u * (B_FULL_V0 + par)), (n >> 1) & 1, abort);
      if (WN > 1) ok = ok && mbar_wait((bar0 + 8u * (B_HALO0 + par)), (n >> 1) & 1, abort);
      ok = ok && mbar_wait((bar0 + 8u * (B_MMA_O0 + par)), (n >> 1) & 1, abort);   // also: every product that reads V is done
      ok = __all_sync(0xffffffffu, ok);
      if (ok && (!GRP || 32 * q4 < valid)) {      // (32 rows behind a partly filled tile's tokens: zeros already)
        tc_fence_after();
        const uint32_t oaddr = tmem + lane_addr + O_COL + 64 * hf;
        float rden[4];
#pragma unroll
        for (int m = 0; m < 4; ++m) {
          // row sum of the masked P + phi(q) . z_prev, both halves gathered by the masking threads
          const float* dr = denbuf + par * 2 * D + 32 * q4 + (lane >> 2) + 8 * m;
          rden[m] = 1.f / (dr[0] + dr[D] + (GRP ? 0.f : eps));  // (three-branch mode: those left the finished factor)
        }
        auto piece = [&](int cc, const uint32_t* f0, const uint32_t* f1) {   // 8 channels: fragments of rows 0-15 and 16-31
          float2 acc[4];
#pragma unroll
          for (int m = 0; m < 4; ++m) {
            const uint32_t* src = (m < 2 ? f0 : f1) + 2 * (m & 1);
            acc[m] = __fmul2_rn(make_float2(__uint_as_float(src[0]), __uint_as_float(src[1])), make_float2(rden[m], rden[m]));
          }
#pragma unroll
          for (int t = 0; t < WN; ++t) {
            uint32_t u[4];
            ldmatrix4(vrow[t] ^ (uint32_t)(cc << 4), u);
            const float2 wt = lds_f2(waddr + t * (D * 4) + cc * 32);
#pragma unroll
            for (int m = 0; m < 4; ++m) acc[m] = __ffma2_rn(wt, bf2(u[m]), acc[m]);
          }
          uint32_t out[4];
#pragma unroll
          for (int m = 0; m < 4; ++m) {
            out[m] = pack2(acc[m].x, acc[m].y);
            // a partly filled tile stays zero below its tokens
            if (GRP && 32 * q4 + (lane >> 2) + 8 * m >= valid) out[m] = 0u;
          }
          stmatrix4(vrow[0] ^ (uint32_t)(cc << 4), out);
        };
        uint32_t a0[16], a1[16];                  // rows 0-15 and 16-31 of 32 channels
        if (!kRollE) {
          LA_TMEM_LD_FRAG4(oaddr, a0);
          LA_TMEM_LD_FRAG4(oaddr + (16u << 16), a1);
        }
#pragma unroll (kRollE ? 1 : 2)
        for (int qq = 0; qq < 2; ++qq) {
          if (kRollE) {
            LA_TMEM_LD_FRAG4(oaddr + 32 * qq, a0);
            LA_TMEM_LD_FRAG4(oaddr + 32 * qq + (16u << 16), a1);
          }
          tmem_wait_ld();
          if (kRollE && qq == 1) {
            tc_fence_before();
            mbar_arrive((bar0 + 8u * (B_EPI0 + par)));         // this accumulator has been read
          }
#pragma unroll
          for (int g = 0; g < 4; ++g) piece(4 * qq + g, a0 + 4 * g, a1 + 4 * g);
          if (!kRollE && qq == 0) {
            LA_TMEM_LD_FRAG4(oaddr + 32, a0);
            LA_TMEM_LD_FRAG4(oaddr + 32 + (16u << 16), a1);
            tmem_wait_ld();
            tc_fence_before();
            mbar_arrive((bar0 + 8u * (B_EPI0 + par)));
          }
        }
      } else {
        mbar_arrive((bar0 + 8u * (B_EPI0 + par)));
      }
      fence_proxy_async();
      mbar_arrive((bar0 + 8u * (B_STAGED0 + par)));
    }
    }
    sync_group_b();                               // both halves of the last halo are complete
    if (fused) cluster_wait();
    if (ok && tid < D && writes_state) {
      // the window to carry on: the last W-1 values of (incoming window ++ this block's v)
      const unsigned char* halo = smem + off_halo(W) + nchunks % 3 * halo_bytes(W);
      for (int i = 0; i < W - 1; ++i)
        win[((size_t)bh * (W - 1) + i) * D + tid] =
            LONG ? halo0[((int)long_taps(W) - W + i) * D + tid]
                 : *reinterpret_cast<const __nv_bfloat16*>(halo + halo_at(i, tid >> 3, W) + (tid & 7) * 2);
      if (tid == 0 && h == 0) pos[bh / H] = (init ? pos[bh / H] : 0) + Ttot;
    }
  }

  // ---- teardown ----
  if (fused && warp >= 16) cluster_wait();        // (groups A and B have waited before they wrote the state)
  tc_fence_before();
  __syncthreads();
  if (sm.abort) {
    if (tid == 0) report(status, LA_ERR_TIMEOUT);
    for (int i = 0; i < 64; ++i) __nanosleep(2000);   // bounded grace period for copies still in flight
  }
  if (warp == kCtrlWarp) {
    __syncwarp();
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(TMEM_COLS) : "memory");
  }
}

// ---- sequence split: local state of a segment ------------------------------------------------------
// For chains too few to fill the GPU the sequence is cut into segments that run as separate CTAs.  This
// kernel computes, for one segment, only its own contribution [dS | dz] = sum phi(k) [v | 1]^T (K and V are
// read, phi applied to K, one product per tile) and stores it in fp32.  In the main pass every segment adds up the
// contributions of those before it.
constexpr int kStateThreads = 288;       // 8 compute warps + 1 issue warp
// (K buffer 1, then V buffer 1 around K buffer 0, V buffer 0 and the ones, which are the third box of both V buffers as
// in the main kernel)
constexpr uint32_t ST_OFF_VQ = TILE_BYTES, ST_OFF_ONES = ST_OFF_VQ + 6 * BOX_BYTES, ST_OFF_SMALL = ST_OFF_ONES + BOX_BYTES;
__host__ __device__ constexpr uint32_t st_kbuf(uint32_t b) { return b ? 0u : ST_OFF_VQ + BOX_BYTES; }
__host__ __device__ constexpr uint32_t st_vbox(uint32_t b, uint32_t half) { return ST_OFF_VQ + (b ? 0u : 4 * BOX_BYTES) + half * vstep(b); }
constexpr uint32_t kStateSmem = ST_OFF_SMALL + 256 + 1024;
// All of them by tile parity: both of the first two tiles may be in place before the issuing lane looks, and both of the last
// two products complete before a compute warp does.
enum { SB_FULL_K0 = 0, SB_FULL_K1, SB_FULL_V0, SB_FULL_V1, SB_PHI0, SB_PHI1, SB_MMA0, SB_MMA1, kStateBars };

template <int PHI>
__global__ void __launch_bounds__(kStateThreads, 1)
segment_state_kernel(const __grid_constant__ CUtensorMap mk, const __grid_constant__ CUtensorMap mv,
                     float* __restrict__ S_out, float* __restrict__ z_out, int* status, int Ttot, int nseg,
                     int seg_len, int nrun, int init, const float* __restrict__ S, const float* __restrict__ z,
                     const __nv_bfloat16* __restrict__ win, __nv_bfloat16* __restrict__ win_copy, int W,
                     const __nv_bfloat16* __restrict__ v_save) {
  extern __shared__ unsigned char smem_dyn[];
  // (an offset into the array rather than an integer cast: the compiler then knows that these are shared-memory
  // addresses: 32-bit arithmetic, ld.shared / st.shared)
  unsigned char* smem = smem_dyn + ((1024u - (smem_u32(smem_dyn) & 1023u)) & 1023u);
  const uint32_t sbase = smem_u32(smem);
  unsigned long long* bars = reinterpret_cast<unsigned long long*>(smem + ST_OFF_SMALL);
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(smem + ST_OFF_SMALL + 128);
  volatile int* abort = reinterpret_cast<int*>(smem + ST_OFF_SMALL + 132);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  // The launch visits the first nrun of a chain's nseg segments (all of them, or all but the last, whose sums no
  // other segment starts from); results go to slot bh * nseg + segment.
  const int bh = blockIdx.x / nrun, sg = blockIdx.x % nrun, u = bh * nseg + sg;
  const int y0 = sg * seg_len, T = min(seg_len, Ttot - y0);
  const int nchunks = (T + TILE - 1) / TILE;
  const uint32_t bar0 = smem_u32(&bars[0]);       // barrier i lives at bar0 + 8 i

  if (tid == 0) {
    for (int i = 0; i < 4; ++i) mbar_init((bar0 + 8u * (i)), 1);
    mbar_init((bar0 + 8u * (SB_PHI0)), 256);
    mbar_init((bar0 + 8u * (SB_PHI1)), 256);
    mbar_init((bar0 + 8u * (SB_MMA0)), 1);
    mbar_init((bar0 + 8u * (SB_MMA1)), 1);
    *abort = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 8) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)), "r"(256u)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  for (int idx = tid; idx < (int)BOX_BYTES / 16; idx += kStateThreads)
    reinterpret_cast<uint4*>(smem + ST_OFF_ONES)[idx] = make_uint4(0u, 0u, 0u, 0u);
  pdl_wait();                                     // everything above touched shared memory and TMEM only
  pdl_trigger();
  __syncthreads();
  if (tid < TILE) *reinterpret_cast<__nv_bfloat16*>(smem + ST_OFF_ONES + swz(tid, 0)) = __float2bfloat16_rn(1.f);
  fence_proxy_async();
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;
  constexpr uint32_t SCOL = 0, ZCOL = 128;

  if (warp == 8) {
    if (lane == 0) {
      auto load_tile = [&](int n) {
        const uint32_t b2 = n & 1;
        mbar_expect_tx((bar0 + 8u * (SB_FULL_K0 + b2)), TILE_BYTES);
        tma_load(sbase + st_kbuf(b2), &mk, 0, y0 + n * TILE, bh, (bar0 + 8u * (SB_FULL_K0 + b2)));
        tma_load(sbase + st_kbuf(b2) + BOX_BYTES, &mk, 64, y0 + n * TILE, bh, (bar0 + 8u * (SB_FULL_K0 + b2)));
        mbar_expect_tx((bar0 + 8u * (SB_FULL_V0 + b2)), TILE_BYTES);
        tma_load(sbase + st_vbox(b2, 0), &mv, 0, y0 + n * TILE, bh, (bar0 + 8u * (SB_FULL_V0 + b2)));
        tma_load(sbase + st_vbox(b2, 1), &mv, 64, y0 + n * TILE, bh, (bar0 + 8u * (SB_FULL_V0 + b2)));
      };
      for (int n = 0; n < 2 && n < nchunks; ++n) load_tile(n);
      for (int n = 0; n < nchunks; ++n) {
        const uint32_t b2 = n & 1;
        if (!mbar_wait((bar0 + 8u * (SB_PHI0 + b2)), (n >> 1) & 1, abort) || !mbar_wait((bar0 + 8u * (SB_FULL_V0 + b2)), (n >> 1) & 1, abort)) break;
        tc_fence_after();
        const uint32_t k_mn = desc_lo(sbase + st_kbuf(b2), BOX_BYTES), v_mn = desc_lo(sbase + st_vbox(b2, 0), vstep(b2));
#pragma unroll
        for (int ks = 0; ks < 8; ++ks)       // [dS | dz] += phi(K)^T [V | 1]
          mma_bf16(tmem + SCOL, desc64(k_mn + kstep_mnmajor(ks)), desc64(v_mn + kstep_mnmajor(ks)), idesc(true, true, 144),
                   n > 0 || ks > 0);
        mma_commit((bar0 + 8u * (SB_MMA0 + b2)));
        if (!mbar_wait((bar0 + 8u * (SB_MMA0 + b2)), (n >> 1) & 1, abort)) break;       // both buffers of this tile are free
        if (n + 2 < nchunks) load_tile(n + 2);
      }
    }
  } else {
    bool ok = true;
    for (int n = 0; n < nchunks; ++n) {
      const int valid = min(TILE, T - n * TILE);
      ok = ok && mbar_wait((bar0 + 8u * (SB_FULL_K0 + (n & 1))), (n >> 1) & 1, abort);
      ok = __all_sync(0xffffffffu, ok);
      if (ok) {
        const int ct = tid & 15, rg = tid >> 4;
        unsigned char* Kb = smem + st_kbuf(n & 1) + (ct >> 3) * BOX_BYTES;
        uint4 x[8];                                             // all eight loads first: they do not wait for the stores
#pragma unroll
        for (int i = 0; i < 8; ++i) x[i] = *reinterpret_cast<const uint4*>(Kb + swz(rg + 16 * i, ct & 7));
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          const int j = rg + 16 * i;
          *reinterpret_cast<uint4*>(Kb + swz(j, ct & 7)) = j < valid ? phi8<PHI>(x[i]) : make_uint4(0u, 0u, 0u, 0u);
        }
      }
      if (valid < TILE && y0 + T < Ttot) {          // rows of the next segment: zeros (0 times a v that is not finite is not 0)
        ok = ok && mbar_wait((bar0 + 8u * (SB_FULL_V0 + (n & 1))), (n >> 1) & 1, abort);
        ok = __all_sync(0xffffffffu, ok);
        if (ok)
          for (int idx = tid; idx < (TILE - valid) * 16; idx += 256)
            *reinterpret_cast<uint4*>(smem + st_vbox(n & 1, (idx & 15) >> 3) + swz(valid + (idx >> 4), idx & 7)) = make_uint4(0u, 0u, 0u, 0u);
      }
      fence_proxy_async();
      mbar_arrive((bar0 + 8u * (SB_PHI0 + (n & 1))));
    }
    const int l = nchunks - 1;                      // (its barrier is at most one phase behind here: tile l was loaded only after
                                                    // product l - 2 had completed)
    ok = ok && mbar_wait((bar0 + 8u * (SB_MMA0 + (l & 1))), (l >> 1) & 1, abort);
    ok = __all_sync(0xffffffffu, ok);
    if (ok) {
      tc_fence_after();
      const int r = 32 * (warp & 3) + lane, hf = warp >> 2;
      const uint32_t lane_addr = (uint32_t)(32 * (warp & 3)) << 16;
      // Where the chain continues a state, its first segment adds that state to its sums and leaves a copy (with the
      // window) for the main pass, whose last segments overwrite the caller's.
      const bool base = init && sg == 0;
      const size_t copy = (size_t)bh * nseg + nseg - 1;
      const size_t at = (size_t)(32 * (warp & 3) + (lane >> 2)) * D + 64 * hf + 2 * (lane & 3);
#pragma unroll
      for (int i = 0; i < 2; ++i) {                 // rows 16 i ... 16 i + 15 of this warp's 32
        uint32_t v[32], x[32];
        if (base) frag_load(S + (size_t)bh * D * D + at + 16 * i * D, x);
        LA_TMEM_LD_FRAG8(tmem + lane_addr + ((uint32_t)(16 * i) << 16) + SCOL + 64 * hf, v);
        tmem_wait_ld();
        if (base) {
          frag_store(S_out + copy * D * D + at + 16 * i * D, x);
          frag_add(v, x);
        }
        frag_store(S_out + (size_t)u * D * D + at + 16 * i * D, v);
      }
      if (hf == 0) {
        const uint32_t zz = tmem_ld1(tmem + lane_addr + ZCOL);
        tmem_wait_ld();
        float x = __uint_as_float(zz);
        if (base) {
          const float c = z[(size_t)bh * D + r];
          z_out[copy * D + r] = c;
          x += c;
        }
        z_out[(size_t)u * D + r] = x;
      }
      if (base)
        for (int idx = tid; idx < (W - 1) * D; idx += 256)
          win_copy[(size_t)bh * (W - 1) * D + idx] = win[(size_t)bh * (W - 1) * D + idx];
      // Where the outputs take the place of v: the rows that the next segment's window reaches back to.
      if (v_save) {
        const size_t chains = gridDim.x / nrun, from = ((size_t)bh * Ttot + y0 + T - (W - 1)) * D;
        for (int idx = tid; idx < (W - 1) * D; idx += 256)
          win_copy[(chains + (size_t)bh * (nseg - 1) + sg) * (W - 1) * D + idx] = v_save[from + idx];
      }
    }
  }
  tc_fence_before();
  __syncthreads();
  if (*abort) {
    if (tid == 0) report(status, LA_ERR_TIMEOUT);
    for (int i = 0; i < 64; ++i) __nanosleep(2000);
  }
  if (warp == 8) {
    __syncwarp();
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(256u) : "memory");
  }
}

// The sums of the segments 0 ... s of a chain into slot s, in place (s < nseg - 1).
// grid = (BH, d*d / 1024), 256 threads, four consecutive elements of S per thread; loads in batches of sixteen slots, all
// in flight at once, only the additions are sequential.
__global__ void __launch_bounds__(256)
prefix_kernel(float* __restrict__ S_seg, float* __restrict__ z_seg, int nseg) {
  const int bh = blockIdx.x, e4 = (blockIdx.y * 256 + threadIdx.x) * 4;
  pdl_wait();
  pdl_trigger();
  float* Sp = S_seg + (size_t)bh * nseg * D * D + e4;
  float4 run = make_float4(0.f, 0.f, 0.f, 0.f);
  for (int s0 = 0; s0 < nseg - 1; s0 += 16) {
    float4 d[16];
#pragma unroll
    for (int j = 0; j < 16; ++j)
      if (s0 + j < nseg - 1) d[j] = *reinterpret_cast<const float4*>(Sp + (size_t)(s0 + j) * D * D);
#pragma unroll
    for (int j = 0; j < 16; ++j)
      if (s0 + j < nseg - 1) {
        run.x += d[j].x, run.y += d[j].y, run.z += d[j].z, run.w += d[j].w;
        *reinterpret_cast<float4*>(Sp + (size_t)(s0 + j) * D * D) = run;
      }
  }
  if (blockIdx.y == 0 && threadIdx.x < D) {
    float* zp = z_seg + (size_t)bh * nseg * D + threadIdx.x;
    float rz = 0.f;
    for (int s0 = 0; s0 < nseg - 1; s0 += 16) {
      float d[16];
#pragma unroll
      for (int j = 0; j < 16; ++j)
        if (s0 + j < nseg - 1) d[j] = zp[(size_t)(s0 + j) * D];
#pragma unroll
      for (int j = 0; j < 16; ++j)
        if (s0 + j < nseg - 1) zp[(size_t)(s0 + j) * D] = rz += d[j];
    }
  }
}

// ---- host side -------------------------------------------------------------------------------------
typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

static EncodeTiledFn encode_fn() {
  static EncodeTiledFn fn = [] {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &p, cudaEnableDefault, &q) != cudaSuccess ||
        q != cudaDriverEntryPointSuccess)
      p = nullptr;
    return reinterpret_cast<EncodeTiledFn>(p);
  }();
  return fn;
}

// [BH, T, 128] bf16 viewed as a 3-D tensor; boxes of 64 columns x 128 rows x 1, 128-byte swizzle.
// Rows past T read as zeros and are clipped on store.
static bool make_map(CUtensorMap* m, const void* base, int BH, int T, int box_rows = TILE) {
  EncodeTiledFn fn = encode_fn();
  if (!fn) return false;
  cuuint64_t dims[3] = {(cuuint64_t)D, (cuuint64_t)T, (cuuint64_t)BH};
  cuuint64_t strides[2] = {(cuuint64_t)D * 2, (cuuint64_t)T * D * 2};
  cuuint32_t box[3] = {64, (cuuint32_t)box_rows, 1};
  cuuint32_t es[3] = {1, 1, 1};
  return fn(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void*>(base), dims, strides, box, es,
            CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

}  // namespace tc

// What the chains of a launch start from and how they are cut (one piece per chain: everything null).
struct Split {
  int nseg = 1, seg_len = 0;
  float *S = nullptr, *z = nullptr;
  const __nv_bfloat16* win = nullptr;
  int prefixed = 0;
  int fused = 0;      // one cluster per chain, whose blocks form the segments' sums themselves
  int saved = 0;      // the rows of v before each segment have been copied to the workspace
};

template <int PHI>
static cudaError_t launch_w(la_ctx* ctx, int BH, int T, const CUtensorMap& mq, const CUtensorMap& mk, const CUtensorMap& mv,
                            const CUtensorMap& mo, const void* v, const float* w, int init, const la_state& st,
                            const Split& sp, cudaStream_t s, bool grouped = false, float alpha = 1.f, float sm_scale = 1.f,
                            int tstep = tc::TILE, int gsz = 0) {
  const la_config& c = ctx->cfg;
  const bool lng = tc::long_epilogue(c.conv_taps, grouped);
  const size_t smem = grouped ? tc::smem_bytes_grp(c.conv_taps, lng) : lng ? tc::smem_bytes_long(c.conv_taps, false) : tc::smem_bytes(c.conv_taps);
  auto kern = tc::prefill_tc_kernel<PHI, 3>;
  if (grouped) {
    kern = gsz ? (lng ? tc::prefill_tc_kernel<PHI, -1, 2> : tc::prefill_tc_kernel<PHI, 3, 2>)
               : (lng ? tc::prefill_tc_kernel<PHI, -1, 1> : tc::prefill_tc_kernel<PHI, 3, 1>);
  } else
  switch (c.conv_taps) {     // short windows: the tap loop unrolled; the others: the long epilogue
    case 1: kern = tc::prefill_tc_kernel<PHI, 1>; break;
    case 2: kern = tc::prefill_tc_kernel<PHI, 2>; break;
    case 3: kern = tc::prefill_tc_kernel<PHI, 3>; break;
    case 4: kern = tc::prefill_tc_kernel<PHI, 4>; break;
    case 5: kern = tc::prefill_tc_kernel<PHI, 5>; break;
    case 6: case 7: case 8: kern = tc::prefill_tc_kernel<PHI, -1>; break;
    default: kern = tc::prefill_tc_kernel<PHI, -2>; break;
  }
  cudaError_t e = allow_smem((const void*)kern, ctx->device);
  if (e != cudaSuccess) return e;
  ctx->launches += 1;
  const int units = BH * sp.nseg;
  // Programmatic dependent launch where this launch and the one behind it fit on the SMs together (that one's set-up then
  // runs beside this one's tiles), and behind the pre-pass.  Not for fuller grids: the blocks that start early take the
  // SMs that the launch before left idle (128 chains of 2048 tokens, 3 taps: 70 against 65 us).
  const int early = 2 * units <= ctx->sm_count;
  return launch_cluster(sp.fused ? sp.nseg : 1, early || sp.nseg > 1, kern, dim3(units), dim3(tc::kThreads), smem, s, mq, mk, mv, mo, w, st.S, st.z,
                          (__nv_bfloat16*)st.win, st.pos, ctx->d_status, c.H, T, c.conv_taps, c.eps, init, sp.nseg,
                          sp.nseg > 1 ? sp.seg_len : T, sp.S, sp.z, sp.win, sp.prefixed, sp.fused, sp.saved ? sp.win + (size_t)BH * (c.conv_taps - 1) * tc::D : (const __nv_bfloat16*)v,
                          sp.saved ? (sp.nseg - 1) * (c.conv_taps - 1) : T, sp.saved ? c.conv_taps - 1 : sp.seg_len, alpha,
                          sm_scale, tstep, gsz, early);
}
static cudaError_t launch_phi(la_ctx* ctx, int BH, int T, const CUtensorMap& mq, const CUtensorMap& mk, const CUtensorMap& mv,
                              const CUtensorMap& mo, const void* v, const float* w, int init, const la_state& st,
                              const Split& sp, cudaStream_t s, bool grouped = false, float alpha = 1.f, float sm_scale = 1.f,
                              int tstep = tc::TILE, int gsz = 0) {
  return ctx->cfg.phi == LA_PHI_ELU1
             ? launch_w<LA_PHI_ELU1>(ctx, BH, T, mq, mk, mv, mo, v, w, init, st, sp, s, grouped, alpha, sm_scale, tstep, gsz)
             : launch_w<LA_PHI_RELU>(ctx, BH, T, mq, mk, mv, mo, v, w, init, st, sp, s, grouped, alpha, sm_scale, tstep, gsz);
}

// Segments per chain for a launch of BH chains of T tokens: 1 unless the chains are too few to fill the GPU and
// long enough to cut (every segment a whole number of tiles).
constexpr int kSplitMinTiles = 6;
// Up to this many segments per chain the blocks of the main pass add up the sums before them as they load their state;
// beyond it a launch of its own forms the prefixes.  (Reached where clusters of that many are not all resident, as with 46 to
// 49 chains in 3 segments: 900 tokens 28.0 us in place, 30.6 with the launch; 2000 tokens 47.0 and 48.5.)
constexpr int kSumInPlace = 4;
static void plan_split(const la_ctx* ctx, int BH, int T, int* nseg, int* seg_len, int tile = tc::TILE) {
  *nseg = 1;
  *seg_len = T;
  int tiles = (T + tc::TILE - 1) / tc::TILE;
  if (2 * BH > ctx->sm_count || tiles < kSplitMinTiles) return;
  // One wave of thread blocks: as many segments per chain as fit on the SMs at once.  (Measured on 32 chains of
  // 32768 tokens: 4 segments per chain 418 us, 9 segments (two waves) 432 us, 13: 456, 18: 483 -- a second wave
  // never fills as well as the first, and every segment costs a 64 KB state written and read back.)
  int n = std::min(ctx->sm_count / BH, tiles), per = (tiles + n - 1) / n;
  n = (tiles + per - 1) / per;
  // Shorter tiles (of the three-branch block) are shared out over at most as many segments: rounded on their own they could
  // make more (8 chains of 2306 tokens: 10 segments of 128-token tiles, 13 of 96), and the caller's workspace, whose size is
  // asked for without a group, would be too small.
  tiles = (T + tile - 1) / tile;
  per = (tiles + n - 1) / n;
  n = (tiles + per - 1) / per;
  if (n < 2) return;
  *nseg = n;
  *seg_len = per * tile;
}
// `rows`: with room for the W - 1 rows of v before each segment but the first.
static size_t split_bytes(const la_config& c, int BH, int nseg, bool rows) {
  return (size_t)BH * ((size_t)nseg * (tc::D * tc::D + tc::D) * 4 + (size_t)(c.conv_taps > 1 ? c.conv_taps - 1 : 1) * tc::D * 2 +
                       (rows ? (size_t)(nseg - 1) * (c.conv_taps - 1) * tc::D * 2 : 0));
}

size_t prefill_workspace_bytes(const la_ctx* ctx, int B, int T) {
  const la_config& c = ctx->cfg;
  if (c.io_dtype != LA_BF16 || c.d != tc::D) return 0;
  int nseg, seg_len;
  plan_split(ctx, B * c.H, T, &nseg, &seg_len);
  return nseg > 1 ? split_bytes(c, B * c.H, nseg, true) : 0;
}

// How many clusters of n blocks, one block per SM, the device holds at once.
constexpr int kMaxCluster = 8;
static int resident_clusters(la_ctx* ctx, int n) {
  if (ctx->max_clusters[n] == 0) {
    auto kern = tc::prefill_tc_kernel<LA_PHI_ELU1, 3>;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(n);
    cfg.blockDim = dim3(tc::kThreads);
    cfg.dynamicSmemBytes = tc::kMaxSmem;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = n;
    attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    int got = 0;
    if (allow_smem((const void*)kern, ctx->device) != cudaSuccess ||
        cudaOccupancyMaxActiveClusters(&got, kern, &cfg) != cudaSuccess) {
      cudaGetLastError();
      got = 0;
    }
    ctx->max_clusters[n] = got > 0 ? got : -1;
  }
  return ctx->max_clusters[n];
}

// Cuts the chains where that pays and the workspace allows it: launches what forms the segments' starting states.  `tile`:
// tokens per tile of the main pass; mk, mv: maps with boxes of 128 rows.
static cudaError_t launch_split(la_ctx* ctx, int BH, int T, int tile, const CUtensorMap& mk, const CUtensorMap& mv, int init,
                                const la_state& st, const void* v, const void* o, Split* out, cudaStream_t s) {
  Split& sp = *out;
  const la_config& c = ctx->cfg;
  plan_split(ctx, BH, T, &sp.nseg, &sp.seg_len, tile);
  if (sp.nseg > 1 && (ctx->ws == nullptr || T < c.conv_taps)) sp = Split();
  const bool fits = sp.nseg > 1 && sp.nseg <= kMaxCluster && BH <= resident_clusters(ctx, sp.nseg);   // one cluster per chain
  // Outputs in the place of v: the blocks of a cluster read the rows before their segments ahead of a barrier that every store is
  // behind; in a grid without one they would race with the stores of the segment before, so copies are made first.
  const uintptr_t va = (uintptr_t)v, oa = (uintptr_t)o, bytes = (uintptr_t)BH * T * tc::D * 2;
  const bool save = !fits && c.conv_taps > 1 && va < oa + bytes && oa < va + bytes;
  if (sp.nseg > 1 && ctx->ws_bytes < split_bytes(c, BH, sp.nseg, save)) sp = Split();
  if (sp.nseg > 1) {
    // Sequence split: the sums of all segments but the last, then every segment as its own CTA.
    const int nseg = sp.nseg, units = BH * nseg;
    float* S_seg = static_cast<float*>(ctx->ws);
    float* z_seg = S_seg + (size_t)units * tc::D * tc::D;
    __nv_bfloat16* win_seg = reinterpret_cast<__nv_bfloat16*>(z_seg + (size_t)units * tc::D);
    sp.S = S_seg, sp.z = z_seg, sp.win = win_seg;
    // Up to 8 segments (a portable cluster): one launch, provided that all the clusters are resident at once.  (32 chains of
    // 1700 tokens, 4 segments each: 40.7 us with the sums formed by a launch of their own, 37 so; 32 x 3000: 55 and
    // 50; 32 x 32768 no difference.)
    if (fits) {
      sp.fused = 1;
      return cudaSuccess;
    }
    auto skern = c.phi == LA_PHI_ELU1 ? tc::segment_state_kernel<LA_PHI_ELU1> : tc::segment_state_kernel<LA_PHI_RELU>;
    cudaError_t e = allow_smem((const void*)skern, ctx->device);
    if (e != cudaSuccess) return e;
    ctx->launches += 1;
    e = launch_pdl(skern, dim3(BH * (nseg - 1)), dim3(tc::kStateThreads), tc::kStateSmem, s, mk, mv, S_seg, z_seg,
                         ctx->d_status, T, nseg, sp.seg_len, nseg - 1, init, (const float*)st.S, (const float*)st.z,
                         (const __nv_bfloat16*)st.win, win_seg, c.conv_taps, save ? (const __nv_bfloat16*)v : nullptr);
    sp.saved = save;
    if (e != cudaSuccess) return e;
    if (nseg > kSumInPlace) {
      sp.prefixed = 1;
      ctx->launches += 1;
      e = launch_pdl(tc::prefix_kernel, dim3(BH, tc::D * tc::D / 1024), dim3(256), 0, s, S_seg, z_seg, nseg);
      if (e != cudaSuccess) return e;
    }
  }
  return cudaSuccess;
}

cudaError_t launch_prefill_tc(la_ctx* ctx, int B, int T, const void* q, const void* k, const void* v, const float* w,
                              int init, const la_state& st, void* o, cudaStream_t s, bool* handled) {
  const la_config& c = ctx->cfg;
  *handled = false;
  if (c.io_dtype != LA_BF16 || c.d != tc::D) return cudaSuccess;
  if ((tc::long_epilogue(c.conv_taps) ? tc::smem_bytes_long(c.conv_taps, false) : tc::smem_bytes(c.conv_taps)) > tc::kMaxSmem)
    return cudaSuccess;                                                  // (does not happen up to LA_MAX_TAPS)
  const int BH = B * c.H;
  CUtensorMap mq, mk, mv, mo;
  if (!tc::make_map(&mq, q, BH, T) || !tc::make_map(&mk, k, BH, T) || !tc::make_map(&mv, v, BH, T) ||
      !tc::make_map(&mo, o, BH, T))
    return cudaErrorNotSupported;   // the driver cannot encode tensor maps: reported, never a silent slow path
  *handled = true;
  Split sp;
  const cudaError_t e = launch_split(ctx, BH, T, tc::TILE, mk, mv, init, st, v, o, &sp, s);
  if (e != cudaSuccess) return e;
  return launch_phi(ctx, BH, T, mq, mk, mv, mo, v, w, init, st, sp, s);
}

// The three-branch block on the tensor cores: bf16 io, d = 128, groups of 32 to 128 tokens (groups of 32 and 64 share
// tiles of 128; any other has a tile of its own, partly filled, which still beats the CUDA-core kernel several times;
// below 32 that kernel takes over), and few enough taps for the 4 KB of extra shared memory.  Sets *handled to false
// otherwise (the CUDA-core kernel takes those).
cudaError_t launch_prefill_grouped_tc(la_ctx* ctx, int B, int T, const void* q, const void* k, const void* v, const float* w,
                                      int group, float alpha, float scale, int init, const la_state& st, void* o,
                                      cudaStream_t s, bool* handled) {
  const la_config& c = ctx->cfg;
  *handled = false;
  if (c.io_dtype != LA_BF16 || c.d != tc::D || group < 32 || group > tc::TILE) return cudaSuccess;
  if (tc::smem_bytes_grp(c.conv_taps, tc::long_epilogue(c.conv_taps, true)) > tc::kMaxSmem) return cudaSuccess;
  const int BH = B * c.H;
  const int gsz = group == 32 || group == 64 ? group : 0, tile = gsz ? tc::TILE : group;
  CUtensorMap mq, mk, mv, mo, mk1, mv1;
  if (!tc::make_map(&mq, q, BH, T, tile) || !tc::make_map(&mk, k, BH, T, tile) || !tc::make_map(&mv, v, BH, T, tile) ||
      !tc::make_map(&mo, o, BH, T, tile) || (tile != tc::TILE && (!tc::make_map(&mk1, k, BH, T) || !tc::make_map(&mv1, v, BH, T))))
    return cudaErrorNotSupported;
  *handled = true;
  Split sp;
  const cudaError_t e = launch_split(ctx, BH, T, tile, tile != tc::TILE ? mk1 : mk, tile != tc::TILE ? mv1 : mv, init, st, v, o, &sp, s);
  if (e != cudaSuccess) return e;
  return launch_phi(ctx, BH, T, mq, mk, mv, mo, v, w, init, st, sp, s, true, alpha, scale, tile, gsz);
}

// The sums of one segment on the tensor cores (bf16 io, d = 128): the kernel of the sequence split with one segment
// per (batch, head) chain.
cudaError_t launch_segment_state_tc(la_ctx* ctx, int B, int T, const void* k, const void* v, float* dS, float* dz,
                                    cudaStream_t s, bool* handled) {
  const la_config& c = ctx->cfg;
  *handled = false;
  if (c.io_dtype != LA_BF16 || c.d != tc::D) return cudaSuccess;
  const int BH = B * c.H;
  CUtensorMap mk, mv;
  if (!tc::make_map(&mk, k, BH, T) || !tc::make_map(&mv, v, BH, T)) return cudaErrorNotSupported;
  auto skern = c.phi == LA_PHI_ELU1 ? tc::segment_state_kernel<LA_PHI_ELU1> : tc::segment_state_kernel<LA_PHI_RELU>;
  *handled = true;
  cudaError_t e = allow_smem((const void*)skern, ctx->device);
  if (e != cudaSuccess) return e;
  ctx->launches += 1;
  return launch_cluster(1, false, skern, dim3(BH), dim3(tc::kStateThreads), tc::kStateSmem, s, mk, mv, dS, dz, ctx->d_status, T,
                          1, T, 1, 0, (const float*)nullptr, (const float*)nullptr, (const __nv_bfloat16*)nullptr,
                          (__nv_bfloat16*)nullptr, c.conv_taps, (const __nv_bfloat16*)nullptr);
}

}  // namespace la
