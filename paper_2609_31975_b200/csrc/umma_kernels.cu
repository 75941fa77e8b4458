// Batched path on the 5th-generation tensor cores (tcgen05.mma, accumulators in TMEM), bf16 storage.
//
//   umma_rows_kernel<GATE>  Z[H, B] = W[H, K] X[B, K]^T + bias (+ fixed-matrix term), activation, gate values,
//                           "any token fires" bit per neuron             (Eq. 1 gate / LoPA U and V stages, batched)
//   umma_rows_kernel<UP>    compacts those bits into the union list of fired neurons (Sec. 5.4), then over that
//                           list: Up = W_up[idx] X^T, Hm = a . A_3(Up), stored as bf16 HmT[b][u]
//   umma_down_kernel        y[b][d] = sum over the list rows u of HmT[b][u] W_down[idx[u]][d]
//   rmsnorm_split_kernel    LoPA: n = RMSNorm(v) as bf16 high / low pairs (the B operand of the U stage)
//
// Rows kernels: one CTA owns a tile of up to 128 weight rows (TMEM lanes) x Npad token columns (Npad = columns
// rounded up to 16); tiles of up to 64 rows use M = 64:
//   warps 0-3  producers: TMA tensor-map copies bring the tile's weight rows and the Npad token rows of a stage's
//              64-wide K blocks into the 128-byte-swizzled K-major layout the tensor core reads (mbarrier
//              complete_tx).  Gate: one tiled copy of the tile's consecutive rows per block.  Union rows:
//              tile::gather4, each lane of the warp fetching four listed rows.
//   warps 8-11 one thread each issues tcgen05.mma (N=Npad, K=16, four per K block) for "its" ring slots into an
//              accumulator of its own and commits each stage's completion to the "slot free" mbarrier.  The serial
//              wait - issue - commit chain of one thread takes on the order of a thousand cycles per stage whatever
//              the MMA shape, so several issuers (four when the ring divides evenly among them, else two) are what
//              lets the copies run at memory speed; warp 8 allocates and frees the TMEM columns
//   warps 4-7  epilogue: tcgen05.ld the accumulator row of "their" neuron (all accumulators added), apply the
//              gate / scale epilogue; for wide batches all twelve warps share the epilogue of the CTA's last tile
// A problem of up to 256 rows per SM is cut into one or two tiles per SM, all of one height, but short rows and most wide
// batches over more than 128 into tiles of 128 (see tile_rows_for).  The ring of
// stages (up to 12) is cut out of the dynamic shared memory on the device, once the tile height is known.
// Every kernel here is launched with programmatic dependent launch: set-up first, griddepcontrol.wait before the
// first dependent read or global write.
// Weight-only int8 / int4 rows (QB = 8 / 4): the copies bring the codes (and the token rows) into the ring slots;
// four more warps (the last four of the CTA, two pairs that alternate over the stages) expand the codes to bf16 --
// every code is an integer bf16 holds exactly -- in the swizzled layout, into a short ring of expanded blocks of
// its own (rows kernels; down kernel, where that leaves more slots for the copies) or the slot's block area, and
// arrive on a "ready" barrier that the MMA issuers wait for instead of "full"; the row scales are applied to the
// accumulator rows in the epilogue (the down projection's are folded into Hm).  With the weights as the A operand
// the tensor core takes 32 bytes of bf16 per cycle and SM whatever the token count, i.e. 16 codes per cycle:
// quantised batches are bound by that rate, not by their bytes.
// Up to 256 token columns go through in one pass.  Wide batches (npad > 128) leave room for two accumulators and a ring
// of four stages of ~40 KB (two with expanded codes and 241 columns or more), too few for the token rows that every CTA reads again
// (200 tokens x 4096: 1.6 MB a CTA through L2 beside 0.8 MB of weights).  There the rows kernels run in pairs of CTAs that hold half
// of the token rows each (PAIR, see umma_rows_pairs).  200 tokens, 4096 x 14336, bf16: 100 us in one pass (short runs), 333 in four.
// Every wait is bounded by a cycle budget; on expiry the status word is set, all roles wind down and the TMEM
// columns are released before the CTA exits.
#include "umma_kernels.cuh"

#include <cuda.h>

#include "common.cuh"
#include "fused_kernel.cuh"
#include "sparse_ffn.h"

namespace sffn {

static_assert(kUmmaActIdentity == kActNone, "identity epilogue code");

namespace {

constexpr int kTileRows = 128;
constexpr int kAtomK = 64;                           // bf16 elements of one 128-byte swizzle row
constexpr int kAAtomBytes = kTileRows * 128;         // 16 KB: one [128 rows x 64 k] swizzled block
constexpr int kThreads = 320;                        // 4 producer warps, 4 epilogue warps, 2 MMA warps
constexpr int kThreadsRows = 384;                    // rows kernels: up to 4 MMA warps
constexpr int kProducerWarps = 4;
constexpr int kMaxStages = 16;                       // barrier slots; bf16 rows use up to 12
constexpr int kMaxStagesBf16 = 12;
constexpr int kExpandSlots = 4;                      // quantised rows: ring of expanded bf16 blocks
constexpr int kDownExpand = 4;                       // the same in the down kernel's, where it has two rings (2 or 4)
constexpr int kWalkMinTokens = 32;                   // batches from which the up kernel may walk every row
constexpr int kWalkAllPercent = 70;                  // union share of the rows from which "every row" is walked
constexpr int kMaxIssuers = 4;
constexpr int kExpandWarps = 4;                      // quantised rows: warps that expand the codes to bf16
constexpr int kMaxOwnTiles = 8;                      // tiles of one CTA whose rows are kept in shared memory
constexpr int kHeaderBytes = 1024 + kMaxOwnTiles * kTileRows * 4;  // barriers + scratch, then the row lists

__device__ __forceinline__ uint32_t smem_u32(const void* p) {
  return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}
__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count));
}
__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ bool mbar_try(uint32_t bar, uint32_t parity) {
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
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity, volatile int* abort_flag, int32_t* status,
                                          long long budget) {
  if (mbar_try(bar, parity)) return true;
  const long long t0 = clock64();
  for (;;) {
#pragma unroll 1
    for (int i = 0; i < 64; ++i)
      if (mbar_try(bar, parity)) return true;
    if (*abort_flag) return false;
    if (clock64() - t0 > budget) {
      *abort_flag = 1;
      atomicExch(status, (int32_t)SFFN_ERR_TIMEOUT);
      return false;
    }
  }
}
__device__ __forceinline__ void named_bar_sync(int id, int threads) {
  asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(threads) : "memory");
}
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

// Shared-memory matrix descriptor: K-major operand, 128-byte swizzle, rows 128 bytes apart, groups of
// eight rows 1024 bytes apart (stride byte offset), descriptor version 1 (Blackwell).
__device__ __forceinline__ uint64_t make_desc(uint32_t smem_addr) {
  uint64_t d = 0;
  d |= (uint64_t)((smem_addr >> 4) & 0x3fff);        // start address, 16-byte units
  d |= (uint64_t)1 << 16;                            // leading byte offset (unused for swizzled K-major)
  d |= (uint64_t)(1024 >> 4) << 32;                  // stride byte offset
  d |= (uint64_t)1 << 46;                            // version
  d |= (uint64_t)2 << 61;                            // SWIZZLE_128B
  return d;
}
// The same for an MN-major operand (here: A[m][k] stored as rows k of 64 contiguous m, 128 bytes each):
// eight k rows form a 1024-byte swizzle atom; `k_group_bytes` apart lie successive groups of eight k rows
// (stride byte offset), `mn_atom_bytes` apart successive blocks of 64 m (leading byte offset).
__device__ __forceinline__ uint64_t make_desc_mn(uint32_t smem_addr, uint32_t mn_atom_bytes, uint32_t k_group_bytes) {
  uint64_t d = 0;
  d |= (uint64_t)((smem_addr >> 4) & 0x3fff);
  d |= (uint64_t)((mn_atom_bytes >> 4) & 0x3fff) << 16;
  d |= (uint64_t)((k_group_bytes >> 4) & 0x3fff) << 32;
  d |= (uint64_t)1 << 46;
  d |= (uint64_t)2 << 61;
  return d;
}
// Instruction descriptor: D fp32, A and B bf16, both K-major, M = m (64 or 128), N = n.
__device__ __forceinline__ uint32_t make_idesc(int n, int m = kTileRows) {
  return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(n >> 3) << 17) | ((uint32_t)(m >> 4) << 24);
}
__device__ __forceinline__ void umma(uint32_t tmem_d, uint64_t adesc, uint64_t bdesc, uint32_t idesc, uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}"
      ::"r"(tmem_d), "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate)
      : "memory");
}
// The same for int8 operands (D int32, A and B signed 8-bit, both K-major; one MMA covers K = 32).
__device__ __forceinline__ uint32_t make_idesc_i8(int n, int m = kTileRows) {
  return (2u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(n >> 3) << 17) | ((uint32_t)(m >> 4) << 24);
}
__device__ __forceinline__ void umma_i8(uint32_t tmem_d, uint64_t adesc, uint64_t bdesc, uint32_t idesc, uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::i8 [%0], %1, %2, %3, p;\n\t}"
      ::"r"(tmem_d), "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate)
      : "memory");
}
// The same three for a pair of CTAs (cta_group::2): one thread of the even CTA issues for both.  A's rows m and m + 128 and B's
// columns n and n + N / 2 are in the two CTAs' shared memory at the same offsets, accumulator rows m and m + 128 in their TMEM;
// the commit arrives at the barrier of that offset in both.
__device__ __forceinline__ void umma_pair(uint32_t tmem_d, uint64_t adesc, uint64_t bdesc, uint32_t idesc, uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n\t}"
      ::"r"(tmem_d), "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate)
      : "memory");
}
__device__ __forceinline__ void umma_pair_i8(uint32_t tmem_d, uint64_t adesc, uint64_t bdesc, uint32_t idesc, uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::2.kind::i8 [%0], %1, %2, %3, p;\n\t}"
      ::"r"(tmem_d), "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate)
      : "memory");
}
__device__ __forceinline__ void umma_commit_pair(uint32_t bar) {
  asm volatile("tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;" ::"r"(bar),
               "h"((uint16_t)3)
               : "memory");
}
__device__ __forceinline__ uint32_t cluster_rank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
__device__ __forceinline__ void cluster_arrive() {
  __syncwarp();
  asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
}
__device__ __forceinline__ void cluster_wait() {
  __syncwarp();
  asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ void cluster_sync() {
  cluster_arrive();
  cluster_wait();
}
// The address, in the cluster's window, of this CTA's shared-memory address in the CTA of rank `rank`.
__device__ __forceinline__ uint32_t map_rank(uint32_t addr, uint32_t rank) {
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
  return r;
}
__device__ __forceinline__ void mbar_arrive_cluster(uint32_t bar) {
  asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void umma_commit(uint32_t bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void tmem_ld8_raw(uint32_t taddr, uint32_t* r) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
               : "r"(taddr));
}
// Eight accumulator columns of this thread's TMEM lane, summed over the `nacc` (1, 2 or 4) accumulators
// that lie `stride` columns apart.
__device__ __forceinline__ void tmem_ld8(uint32_t taddr, int nacc, int stride, float* v) {
  uint32_t r0[8], r1[8], r2[8], r3[8];
  tmem_ld8_raw(taddr, r0);
  if (nacc >= 2) tmem_ld8_raw(taddr + stride, r1);
  if (nacc == 4) {
    tmem_ld8_raw(taddr + 2 * stride, r2);
    tmem_ld8_raw(taddr + 3 * stride, r3);
  }
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    float a = __uint_as_float(r0[i]);
    if (nacc >= 2) a += __uint_as_float(r1[i]);
    if (nacc == 4) a += __uint_as_float(r2[i]) + __uint_as_float(r3[i]);
    v[i] = a;
  }
}

// The same for int32 accumulators (summed exactly).
__device__ __forceinline__ void tmem_ld8_int(uint32_t taddr, int nacc, int stride, int* v) {
  uint32_t r0[8], r1[8], r2[8], r3[8];
  tmem_ld8_raw(taddr, r0);
  if (nacc >= 2) tmem_ld8_raw(taddr + stride, r1);
  if (nacc == 4) {
    tmem_ld8_raw(taddr + 2 * stride, r2);
    tmem_ld8_raw(taddr + 3 * stride, r3);
  }
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    int a = (int)r0[i];
    if (nacc >= 2) a += (int)r1[i];
    if (nacc == 4) a += (int)r2[i] + (int)r3[i];
    v[i] = a;
  }
}

// 16 int32 columns of this thread's lane, summed over the accumulators.
__device__ __forceinline__ void tmem_ld16_int(uint32_t taddr, int nacc, int stride, int* v) {
  uint32_t r[16];
  tmem_ld8_raw(taddr, r);
  tmem_ld8_raw(taddr + 8, r + 8);
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
  for (int i = 0; i < 16; ++i) v[i] = (int)r[i];
#pragma unroll 1
  for (int a = 1; a < nacc; ++a) {
    tmem_ld8_raw(taddr + a * stride, r);
    tmem_ld8_raw(taddr + a * stride + 8, r + 8);
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
    for (int i = 0; i < 16; ++i) v[i] += (int)r[i];
  }
}

// Loads (0 where `on` is false) and stores that a predicate turns off: the epilogues' straight-line code has a dozen of them, and
// a branch around each costs more than the access.
__device__ __forceinline__ float ld_f32_if(const float* p, bool on) {
  float v;
  asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.u32 p, %2, 0;\n\tmov.f32 %0, 0f00000000;\n\t@p ld.global.f32 %0, [%1];\n\t}"
               : "=f"(v) : "l"(p), "r"((uint32_t)on) : "memory");
  return v;
}
__device__ __forceinline__ float ld_bf16_if(const __nv_bfloat16* p, bool on) {
  uint16_t v;
  asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.u32 p, %2, 0;\n\tmov.b16 %0, 0;\n\t@p ld.global.u16 %0, [%1];\n\t}"
               : "=h"(v) : "l"(p), "r"((uint32_t)on) : "memory");
  return __uint_as_float((uint32_t)v << 16);
}
__device__ __forceinline__ void st_f32_if(float* p, float v, bool on) {
  asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.u32 p, %2, 0;\n\t@p st.global.f32 [%0], %1;\n\t}" ::"l"(p), "f"(v), "r"((uint32_t)on) : "memory");
}
__device__ __forceinline__ void st_bf16_if(__nv_bfloat16* p, __nv_bfloat16 v, bool on) {
  asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.u32 p, %2, 0;\n\t@p st.global.b16 [%0], %1;\n\t}" ::"l"(p), "h"(__bfloat16_as_ushort(v)), "r"((uint32_t)on)
               : "memory");
}

// What the products with a token's four limbs (most significant first, 7 bits apart) amount to: i0 + i1 / 128 + i2 / 128^2 +
// i3 / 128^3.
__device__ __forceinline__ float limb_sum(int i0, int i1, int i2, int i3) {
  return ((float)i0 + (float)i1 * 0.0078125f) + ((float)i2 * 6.103515625e-05f + (float)i3 * 4.76837158203125e-07f);
}

__device__ __forceinline__ void mbar_expect_tx(uint32_t bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
// Tiled tensor-map copy: box {64 elements, rows} at (element c0, row c1); out-of-range rows read as zero.
__device__ __forceinline__ void tma_tile_2d(uint32_t dst, const CUtensorMap* map, int c0, int c1, uint32_t bar) {
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];" ::"r"(dst),
      "l"(map), "r"(c0), "r"(c1), "r"(bar)
      : "memory");
}
// The same, and the gather below, for a CTA of a pair: `bar` may be the other CTA's.
__device__ __forceinline__ void tma_tile_2d_pair(uint32_t dst, const CUtensorMap* map, int c0, int c1, uint32_t bar) {
  asm volatile(
      "cp.async.bulk.tensor.2d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];" ::"r"(dst),
      "l"(map), "r"(c0), "r"(c1), "r"(bar)
      : "memory");
}
__device__ __forceinline__ void tma_gather4_pair(uint32_t dst, const CUtensorMap* map, int c0, int r0, int r1, int r2,
                                                 int r3, uint32_t bar) {
  asm volatile(
      "cp.async.bulk.tensor.2d.cta_group::2.shared::cluster.global.tile::gather4.mbarrier::complete_tx::bytes [%0], [%1, {%2, "
      "%3, %4, %5, %6}], [%7];" ::"r"(dst),
      "l"(map), "r"(c0), "r"(r0), "r"(r1), "r"(r2), "r"(r3), "r"(bar)
      : "memory");
}
// Gather copy: four rows r0..r3 (any order) x 64 elements starting at element c0 land as four
// consecutive 128-byte rows at dst (the map's box is {64, 1}).
__device__ __forceinline__ void tma_gather4(uint32_t dst, const CUtensorMap* map, int c0, int r0, int r1, int r2,
                                            int r3, uint32_t bar) {
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.tile::gather4.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, "
      "%4, %5, %6}], [%7];" ::"r"(dst),
      "l"(map), "r"(c0), "r"(r0), "r"(r1), "r"(r2), "r"(r3), "r"(bar)
      : "memory");
}

// Eight 4-bit codes of a word as bf16: o[i] holds codes i and i + 4, which are the halves of one shift and mask.  Under the exponent
// of 128 the nibble ^ 8 reads 136 + code, and 136 is subtracted from both at once.
__device__ __forceinline__ void q4_halves(uint32_t w, uint32_t* o) {
  const __nv_bfloat162 bias = __halves2bfloat162(__ushort_as_bfloat16(0x4308), __ushort_as_bfloat16(0x4308));
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const uint32_t both = ((w >> (4 * i)) & 0x000f000fu) ^ 0x43084308u;
    const __nv_bfloat162 v = __hsub2(*reinterpret_cast<const __nv_bfloat162*>(&both), bias);
    o[i] = *reinterpret_cast<const uint32_t*>(&v);
  }
}

// Expands a block of weight codes to bf16: `raw` holds [rows][64] codes (QB = 8: a byte each, +-127; QB = 4: two's-
// complement nibbles, even column in the low nibble), `dst` (1024-byte aligned) receives [rows][64] bf16 in the
// 128-byte-swizzled K-major layout (16-byte chunk c of row i at i * 128 + ((c ^ (i & 7)) * 16)).  Thread t of nthr
// takes the 16-code quarter t % 4 of rows t / 4, t / 4 + nthr / 4, ... (four of them in flight): a quarter warp reads two whole raw rows
// and writes chunks of two rows that share no bank.  An int8 code c becomes the fp32 2^23 + (c + bias) by a byte
// permute, the bias and 2^23 are subtracted exactly, and the upper half of that fp32 is the bf16.  ALL: rows = nthr, four a thread.
template <int QB, bool ALL = false>
__device__ __forceinline__ void expand_block(uint32_t raw, uint32_t dst, int rows, int t, int nthr) {
  constexpr int kRawRow = 8 * QB;  // bytes of 64 codes
  constexpr int kUnroll = 4;       // rows of one thread in flight
  const int c = t & 3, step = nthr >> 2;
  for (int row0 = t >> 2; row0 < rows; row0 += kUnroll * step) {
    uint32_t w[kUnroll][4];
#pragma unroll
    for (int u = 0; u < kUnroll; ++u) {
      const int row = row0 + u * step;
      const uint32_t src = raw + row * kRawRow + c * (kRawRow / 4);
      w[u][0] = w[u][1] = w[u][2] = w[u][3] = 0;
      if (ALL || row < rows) {
        if (QB == 8) {
          asm volatile("ld.shared.v4.b32 {%0,%1,%2,%3}, [%4];"
                       : "=r"(w[u][0]), "=r"(w[u][1]), "=r"(w[u][2]), "=r"(w[u][3])
                       : "r"(src));
        } else {
          asm volatile("ld.shared.v2.b32 {%0,%1}, [%2];" : "=r"(w[u][0]), "=r"(w[u][1]) : "r"(src));
        }
      }
    }
#pragma unroll
    for (int u = 0; u < kUnroll; ++u) {
      const int row = row0 + u * step;
      if (!ALL && row >= rows) break;
      uint32_t o[8];  // o[i] = codes 2i, 2i+1 of the quarter
      if (QB == 4) {
#pragma unroll
        for (int q = 0; q < 2; ++q) {
          uint32_t h[4];
          q4_halves(w[u][q], h);
          o[4 * q] = __byte_perm(h[0], h[1], 0x5410);
          o[4 * q + 1] = __byte_perm(h[2], h[3], 0x5410);
          o[4 * q + 2] = __byte_perm(h[0], h[1], 0x7632);
          o[4 * q + 3] = __byte_perm(h[2], h[3], 0x7632);
        }
      } else {
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          const uint32_t v = w[u][i >> 1] ^ 0x80808080u;
          const uint32_t lo = __byte_perm(v, 0x4b000000u, (i & 1) ? 0x7442 : 0x7440), hi = __byte_perm(v, 0x4b000000u, (i & 1) ? 0x7443 : 0x7441);
          const float2 f = add2(make_float2(__uint_as_float(lo), __uint_as_float(hi)), make_float2(-8388736.f, -8388736.f));  // 2^23 + 128
          o[i] = __byte_perm(__float_as_uint(f.x), __float_as_uint(f.y), 0x7632);
        }
      }
      const uint32_t drow = dst + row * 128;
      const int sw = row & 7;
      asm volatile("st.shared.v4.b32 [%0], {%1,%2,%3,%4};" ::"r"(drow + (((2 * c) ^ sw) << 4)), "r"(o[0]), "r"(o[1]),
                   "r"(o[2]), "r"(o[3])
                   : "memory");
      asm volatile("st.shared.v4.b32 [%0], {%1,%2,%3,%4};" ::"r"(drow + (((2 * c + 1) ^ sw) << 4)), "r"(o[4]), "r"(o[5]),
                   "r"(o[6]), "r"(o[7])
                   : "memory");
    }
    if (ALL) break;
  }
}
// int4 codes for the down projection, whose columns are the rows m of the MMA and may come in the order of q4_halves, which its
// epilogue undoes: m = 8 k + 2 i + h holds column 8 k + i + 4 h.  64 rows of 64 codes.  (1.4 instructions a code, where fp32 and
// columns in order took 3: 4096 x 14336, 5 / 64 tokens 45.8 / 87.5 -> 45.0 / 83.9 us, 8192 x 24000, 24 tokens 146 -> 139.)
__device__ __forceinline__ int column_of_row(int m) { return (m & ~7) + ((m & 7) >> 1) + ((m & 1) << 2); }
__device__ __forceinline__ void expand_block_q4_mn(uint32_t raw, uint32_t dst, int t) {
  constexpr int kRows = kAtomK, kStep = 32 * kExpandWarps / 2 / 4, kUnroll = kRows / kStep;  // by a pair of warps, all rows in flight
  const int c = t & 3;
  uint32_t w[kUnroll][2];
#pragma unroll
  for (int u = 0; u < kUnroll; ++u)
    asm volatile("ld.shared.v2.b32 {%0,%1}, [%2];" : "=r"(w[u][0]), "=r"(w[u][1]) : "r"(raw + ((t >> 2) + u * kStep) * 32 + c * 8));
#pragma unroll
  for (int u = 0; u < kUnroll; ++u) {
    const int row = (t >> 2) + u * kStep, sw = row & 7;
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      uint32_t o[4];
      q4_halves(w[u][q], o);
      asm volatile("st.shared.v4.b32 [%0], {%1,%2,%3,%4};" ::"r"(dst + row * 128 + (((2 * c + q) ^ sw) << 4)), "r"(o[0]), "r"(o[1]),
                   "r"(o[2]), "r"(o[3])
                   : "memory");
    }
  }
}
// The same for int4 codes on their way to the int8 MMA: `raw` holds [rows][128] nibbles (64 bytes a row), `dst`
// receives [rows][128] bytes, each 16 x its code (the nibble moved to the upper half of the byte: exact, and the factor
// goes into the row scale), in the same swizzled layout.  Thread t takes the 32 codes of quarter t % 4 of its rows: one
// 16-byte load, two 16-byte stores; per word of eight nibbles two masks and two byte permutes.
// kUnroll rows of a thread are in flight.  Tiles of more than 64 rows: eight, which is all that a thread has, one latency for a stage
// instead of one a row (4096 x 14336, 5 / 24 tokens 47.0 / 62.6 -> 45.8 / 61.2 us, 8192 x 24000 102.6 / 149 -> 98.2 / 146; four in
// flight gain a third of that).  Others, a kernel of their own: one, as more code to fetch costs them more (1024 x 3000, tiles of 24
// rows, 5 tokens 23.2 / 23.6), and the LoPA gate, whose few stages come with the code of V x in the caches (4096 x 14336, r = 512, 2
// tokens 36.0 / 37.8).
constexpr int kTallTile = 64;
template <int kUnroll>
__device__ __forceinline__ void expand_block_q4_i8(uint32_t raw, uint32_t dst, int rows, int t, int nthr) {
  const int c = t & 3, step = nthr >> 2;
#pragma unroll 1
  for (int row0 = t >> 2; row0 < rows; row0 += kUnroll * step) {
    uint32_t w[kUnroll][4];
#pragma unroll
    for (int u = 0; u < kUnroll; ++u) {
      const int row = row0 + u * step;
      w[u][0] = w[u][1] = w[u][2] = w[u][3] = 0;
      if (kUnroll == 1 || row < rows)
        asm volatile("ld.shared.v4.b32 {%0,%1,%2,%3}, [%4];" : "=r"(w[u][0]), "=r"(w[u][1]), "=r"(w[u][2]), "=r"(w[u][3]) : "r"(raw + row * 64 + c * 16));
    }
#pragma unroll
    for (int u = 0; u < kUnroll; ++u) {
      const int row = row0 + u * step;
      if (row >= rows) break;
      uint32_t o[8];
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const uint32_t ev = (w[u][i] << 4) & 0xf0f0f0f0u, od = w[u][i] & 0xf0f0f0f0u;  // even / odd columns, times 16
        o[2 * i] = __byte_perm(ev, od, 0x5140);
        o[2 * i + 1] = __byte_perm(ev, od, 0x7362);
      }
      const uint32_t drow = dst + row * 128;
      const int sw = row & 7;
      asm volatile("st.shared.v4.b32 [%0], {%1,%2,%3,%4};" ::"r"(drow + (((2 * c) ^ sw) << 4)), "r"(o[0]), "r"(o[1]),
                   "r"(o[2]), "r"(o[3])
                   : "memory");
      asm volatile("st.shared.v4.b32 [%0], {%1,%2,%3,%4};" ::"r"(drow + (((2 * c + 1) ^ sw) << 4)), "r"(o[4]), "r"(o[5]),
                   "r"(o[6]), "r"(o[7])
                   : "memory");
    }
  }
}
// Makes this thread's shared-memory stores visible to the tensor core's reads.
__device__ __forceinline__ void fence_proxy_async() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }

// Rows per tile of a GEMM over rows of K elements: the row count spread over the whole grid, one tile or two for each CTA (a
// multiple of 8, the swizzle period), so that every SM streams a share.  Two tiles of equal height, not tiles of 128 rows
// whose second wave leaves most SMs idle: 24000 rows are 273 tiles of 88 rows, where 188 of 128 kept 40 of 148 SMs busy in the
// second half (bf16, 5120 x 20000, 2 / 32 tokens: 80.7 / 155 -> 70.5 / 127 us; int4, 8192 x 24000, 64: 484 -> 339).  128
// where a CTA owns more than two, for short rows (the LoPA gate), whose tiles are gone before the imbalance shows (r = 512 /
// 1024: 0 to 1 % faster; r = 1536, and int4 rows of 2048 codes, which are as many bytes as 512 bf16 elements: equal tiles 0 to 3 %
// faster), and for most wide passes: bf16 rows against more than 128 tokens
// are bound by the token rows that every tile reads through L2, and tiles of 128 are fewer.  There equal tiles pay only where
// their stages are enough smaller for more of them in the ring (tiles of 128 / equal ones: 7168 x 20000, 200 tokens, 4 / 6 slots
// 353 / 329 us, 160 tokens, 6 / 6 slots 270 / 287; 8192 x 20000, 256, 4 / 4: 414 / 474; 6144 x 24576, 200, 4 / 4: 324 / 345).
constexpr int kShortRow = 1024;
constexpr int kRowsSmem = 226 * 1024, kRingBytes = kRowsSmem - 1024 - kHeaderBytes;
// The tallest tiles that two equal ones may be, else 128 (over rows of K elements, qbits as in UmmaRowsParams, B tokens).
inline int equal_tiles_max(int K, int qbits, int B) {
  if (K <= kShortRow) return 0;
  if (qbits != 0 || B <= 128) return kTileRows;
  const int cols = (B + 15) / 16 * 16;
  auto slots = [&](int rows) { return kRingBytes / ((rows + cols) * 128) & ~1; };
  return kRingBytes / (128 * (slots(kTileRows) + 2)) - cols;
}
__host__ __device__ inline int tile_rows_for(int n_rows, int grid, int equal_max) {
  const int per_cta = n_rows > kTileRows * grid ? 2 : 1;
  if (n_rows > 2 * kTileRows * grid) return kTileRows;
  const int t = ((n_rows + per_cta * grid - 1) / (per_cta * grid) + 7) & ~7;
  if (per_cta == 2 && t > equal_max) return kTileRows;
  return t < 8 ? 8 : t > kTileRows ? kTileRows : t;
}

__host__ __device__ inline uint32_t tmem_cols_for(int cols) {
  return cols <= 32 ? 32 : cols <= 64 ? 64 : cols <= 128 ? 128 : cols <= 256 ? 256 : 512;
}

// Third tensor map of the up kernel that may walk every row (tiled boxes over all rows); empty otherwise, so
// that the other instantiations keep their two-map signature.
template <bool HAS>
struct WalkMap {
  CUtensorMap m;
  __device__ const CUtensorMap* get() const { return &m; }
};
template <>
struct WalkMap<false> {
  __device__ const CUtensorMap* get() const { return nullptr; }
};

// v rounded to bf16; v keeps the rest.  Nothing is left of an infinite value.
__device__ __forceinline__ __nv_bfloat16 take_bf16(float& v) {
  const __nv_bfloat16 t = __float2bfloat16(v);
  const float f = __bfloat162float(t), rest = v - f;
  v = fabsf(f) < INFINITY ? rest : 0.f;
  return t;
}

// h of a neuron for a token whose gate value is a: one that did not fire adds zero whatever its W_up row holds.
__device__ __forceinline__ float fired_part(float a, float h) { return a == 0.f ? 0.f : h; }

// Exact sums (EX): the tensor cores truncate when they add onto an accumulator, so a sum over K = 2688 comes out low by
// 1e-6 of its typical size, ten times what fp32 rounding leaves.  Here every two MMAs (K = 32) start an accumulator of
// their own; the epilogue warps add a stage's accumulators in fp32 registers, which round to nearest.  An issuer has one
// place in TMEM (the accumulators of one of its stages) and commits once per stage, to the epilogue warps, which give the
// ring slot and then the place back: a commit per K block took twice as long.  Two sets of four epilogue warps share the
// token columns (at most kExactTokens, in up to three terms: kUmmaExactCols columns).  h, and the LoPA vector, enter as
// three bf16 terms (24 bits).  Error from 64 bits 1.1e-7 to 1.6e-7 over 384 to 7808 columns, the single-token kernels'
// 1.2e-7 to 1.7e-7.  Bound by the round trip of a stage through issuer and epilogue: 0.5 us to 1 us per K block, 12 us to 35
// us per kernel more than without (2688 x 7168, 6 / 60 tokens), against token-by-token calls of 97 / 918 us.
constexpr int kExactTokens = kUmmaExactTokens;
constexpr int kExactHalf = kExactTokens / 2;
constexpr int kExactHalfTerms = 24;   // the same for passes whose tokens come in three terms: 40 tokens, in sets of 24 and 16
constexpr int kExactMmas = 2;         // MMAs that share an accumulator
constexpr int kExactPer = kAtomK / 16 / kExactMmas;  // accumulators of a K block
__host__ __device__ constexpr int exact_issuers(int npad) { return npad <= 64 ? 4 : 2; }
// K blocks of a stage, so that a place takes 128 (two issuers: 256) columns
__host__ __device__ constexpr int exact_atoms(int npad) { return npad <= 16 ? 4 : npad <= 32 ? 2 : 1; }

// Adds the accumulators of one stage (npad columns apart: `accs` of them, each of up to three terms `stride` columns apart)
// up and then onto this thread's sums of the token columns [c0, c1), with what those additions round off collected beside
// them (Kahan 1965) for the end, where an infinite sum has no use for it.  Carried into the next addition instead, it would
// have to be tested each time, about 3 % of a call of 2176 x 4608, 37 tokens.
template <int HALF>
__device__ __forceinline__ void add_stage(uint32_t taddr, int accs, int npad, int c0, int c1, int terms, int stride, float* sum, float* low) {
#pragma unroll
  for (int g = 0; g < HALF; g += 16) {
    if (c0 + g < c1) {
      const bool two = g + 8 < HALF && c0 + g + 8 < c1;  // 16 columns or eight
      const uint32_t at = taddr + c0 + g;
      uint32_t r[16];
      float part[16];
      int acc = 1, off = 0;
      tmem_ld8_raw(at, r);
      if (two) tmem_ld8_raw(at + 8, r + 8);
      asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
      for (int q = 0; q < 16; ++q) part[q] = __uint_as_float(r[q]);
#pragma unroll 1
      for (int i = accs * terms - 1; i > 0; --i) {
        if (acc == accs) { acc = 0; off += stride; }
        tmem_ld8_raw(at + acc * npad + off, r);
        if (two) tmem_ld8_raw(at + acc * npad + off + 8, r + 8);
        ++acc;
        asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
        for (int q = 0; q < 16; ++q) part[q] += __uint_as_float(r[q]);
      }
#pragma unroll
      for (int q = 0; q < 16; ++q)
        if (g + q < HALF) {  // (the upper eight are not used where there are none)
          const float t = sum[g + q] + part[q];
          low[g + q] += part[q] - (t - sum[g + q]);
          sum[g + q] = t;
        }
    }
  }
}
template <int HALF>
__device__ __forceinline__ void finish_sums(float* sum, const float* low) {
#pragma unroll
  for (int i = 0; i < HALF; ++i)
    if (fabsf(sum[i]) < INFINITY) sum[i] += low[i];
}
// Meets `threads` threads at named barrier `id`; true for all of them if any of them came with true.
__device__ __forceinline__ bool named_bar_any(int id, int threads, bool v) {
  uint32_t any;
  asm volatile("{\n\t.reg .pred p, q;\n\tsetp.ne.u32 p, %1, 0;\n\tbarrier.cta.red.or.pred q, %2, %3, p;\n\tselp.u32 %0, 1, 0, q;\n\t}"
               : "=r"(any) : "r"(v ? 1u : 0u), "r"(id), "r"(threads) : "memory");
  return any != 0;
}

enum RowsMode { kGate = 0, kUp = 1, kUpMayWalk = 2 };  // kUpMayWalk: wide batches, see walk_all below

template <int MODE, int QB, bool EX = false, bool PAIR = false>
__global__ void __launch_bounds__(kThreadsRows + (EX ? 128 : 0) + ((QB == 8 || QB == 4 || QB == 2 || QB == 3) ? 32 * kExpandWarps : 0), 1) umma_rows_kernel(const UmmaRowsParams p,
                                                                  const __grid_constant__ CUtensorMap map_w,
                                                                  const __grid_constant__ CUtensorMap map_x,
                                                                  const __grid_constant__ WalkMap<MODE == kUpMayWalk> map_t) {
  constexpr bool UP = MODE != kGate;
  static_assert(!(EX && PAIR) && (!PAIR || QB <= 1), "pairs: bf16 rows, or int8 rows against limbs");
  extern __shared__ __align__(1024) unsigned char smem_raw[];
  // carve: stages first (1024-byte aligned), then barriers and control words
  const int npad = p.npad;
  unsigned char* smem = reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
  // header: barriers (for the largest ring) and control words, scan scratch, this CTA's rows of the union
  // list; then the ring of stages, whose geometry is decided below once the tile height is known
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem);
  int* scan_wt = reinterpret_cast<int*>(smem + 512);   // [warps]
  int* rows_sm = reinterpret_cast<int*>(smem + 1024);  // [kMaxOwnTiles][128]
  const uint32_t stage0 = smem_u32(smem) + kHeaderBytes;
  const uint32_t full = smem_u32(bars), empty = smem_u32(bars + kMaxStages);
  const uint32_t acc_full = smem_u32(bars + 2 * kMaxStages), acc_empty = smem_u32(bars + 2 * kMaxStages + 1);
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + 2 * kMaxStages + 2);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
  const uint32_t ready = smem_u32(bars + 2 * kMaxStages + 4);  // quantised rows: slot t of the bf16 ring is written ...
  const uint32_t afree = ready + 8 * kExpandSlots;             // ... and has been read by its MMAs
  // QB = 3: the same for tall tiles (see expand_block_q4_i8).
  constexpr bool kI4 = QB == 2 || QB == 3;
  constexpr int kRawRow = kI4 ? 64 : 8 * QB;                   // bytes of the codes of one K block (as copied)
  // QB = 1: int8 rows and the tokens as int8 limbs (four per token, see token_limbs_kernel) go straight into
  // kind::i8 MMAs with int32 accumulators: nothing to expand, a K block is 128 codes.  QB = 8 / 4: codes expanded
  // to bf16 by four more warps.
  // QB = 2: int4 rows expanded to int8 (16 x the code, a byte each) for the same kind::i8 MMAs.
  constexpr bool kNat = QB == 1 || kI4, kExp = QB == 8 || QB == 4 || kI4, kQ = QB != 0;
  constexpr int kAtomElems = kNat ? 128 : kAtomK;              // elements of one 128-byte swizzle row

  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  // PAIR: the pair's CTAs go through their tiles together (the second one's last tile may not exist); `first` is the even CTA
  const int rank = PAIR ? (int)cluster_rank() : 0, first = (int)blockIdx.x - rank;
  // Gate mode: a second grid dimension cuts K into runs of blocks (see umma_k_splits), the first `longer_runs` of them one block
  // longer; each writes sums of its own, or adds its own to the others'.  (Not a mode of its own: the gate that follows V x finds
  // its code in the caches, without which calls of bf16 rows take 1 us more.)
  constexpr bool kSplits = MODE == kGate && !EX && !PAIR;
  const int kb_first = kSplits ? (int)blockIdx.y * p.run_blocks + min((int)blockIdx.y, p.longer_runs) : 0;
  const int kblocks = kSplits ? p.run_blocks + ((int)blockIdx.y < p.longer_runs) : p.K / kAtomElems;
  float* const a_out = p.a_out + (kSplits ? (size_t)blockIdx.y * p.split_stride : 0);

  // Set-up that needs nothing from earlier kernels runs while the predecessor in the stream finishes.
  pdl_launch_dependents();
  const int max_acc = npad > 128 ? 2 : kMaxIssuers;  // 512 TMEM columns: wide token blocks leave room for two accumulators
  static_assert(!EX || !kNat, "exact sums: bf16 operands");
  const int place_cols = exact_atoms(npad) * kExactPer * npad;  // EX: columns of an issuer's place
  const uint32_t place_full = afree + 8 * kExpandSlots, place_empty = place_full + 8 * kMaxIssuers;
  constexpr int kExpand0 = kThreadsRows + (EX ? 128 : 0);  // first expander thread
  const uint32_t tmem_cols = tmem_cols_for(EX ? exact_issuers(npad) * place_cols : max_acc * npad);
  if (tid == 0) {
    for (int s = 0; s < kMaxStages; ++s) {
      mbar_init(full + 8 * s, 1);  // the producer's expect_tx arrive; the copies complete the bytes
      mbar_init(empty + 8 * s, 1);
    }
    if (kExp)
      for (int t = 0; t < kExpandSlots; ++t) {
        mbar_init(ready + 8 * t, kExpandWarps / 2);
        mbar_init(afree + 8 * t, 1);
      }
    if (EX)
      for (int q = 0; q < kMaxIssuers; ++q) {
        mbar_init(place_full + 8 * q, 1);
        mbar_init(place_empty + 8 * q, 8);  // one arrival per epilogue warp
      }
    mbar_init(acc_empty, PAIR ? 256 : 128);
    *abort_flag = 0;
    asm volatile("prefetch.tensormap [%0];" ::"l"(&map_w) : "memory");
    asm volatile("prefetch.tensormap [%0];" ::"l"(&map_x) : "memory");
  }
  if (warp == 8) {
    if constexpr (PAIR) {
      asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)), "r"(tmem_cols)
                   : "memory");
      asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
    } else {
      asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)), "r"(tmem_cols)
                   : "memory");
      asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
  }
  // The up kernel needs the gate's results from here on.  The gate kernel's tiles depend on nothing but its
  // own arguments, and its weights are parameters: its producers fill the ring before they wait (see below),
  // every other role of it waits just before its first dependent access.
  if (MODE != kGate) pdl_wait();

  // Union rows: either the list is given (idx, count), or every CTA compacts the gate's "fired" bit masks
  // itself.  The gate kernel leaves one 32-bit word per epilogue warp and tile (word 4 * tile + warp, bit =
  // lane = row rows_per_word * warp + lane of the tile, 32 rows per word for M = 128 tiles and pairs, 16 for M = 64); thread t takes
  // the four words of tile t, and a warp scan plus the warps' totals give the list position of their first set bit.
  const bool own_list = UP && p.words_in != nullptr;
  uint32_t bits[4] = {0, 0, 0, 0};
  int fired_here = 0, first_pos = 0;
  int n_rows;
  if (own_list) {
    if (tid < kThreadsRows && 4 * tid < p.n_words) {
      const uint4 w = __ldcg(reinterpret_cast<const uint4*>(p.words_in) + tid);
      bits[0] = w.x; bits[1] = w.y; bits[2] = w.z; bits[3] = w.w;
    }
    fired_here = __popc(bits[0]) + __popc(bits[1]) + __popc(bits[2]) + __popc(bits[3]);
    int incl = fired_here;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      const int t = __shfl_up_sync(0xffffffffu, incl, d);
      if (lane >= d) incl += t;
    }
    if (lane == 31 && warp < kThreadsRows / 32) scan_wt[warp] = incl;
    __syncthreads();
    int before = 0, total = 0;
#pragma unroll
    for (int w = 0; w < kThreadsRows / 32; ++w) {
      const int t = scan_wt[w];
      before += w < warp ? t : 0;
      total += t;
    }
    first_pos = incl - fired_here + before;
    n_rows = total;
  } else {
    n_rows = p.count ? *p.count : p.R;
  }
  // A union that covers most of the rows is cheaper to walk as "every row" with tiled copies (which stream about
  // 1.5x faster than gathered rows) than as a list: unfired rows have a = 0 for every token, so their h is 0.
  // The list and its length are still published; the down kernel is told through *walk_all to do the same.
  const int n_listed = n_rows;
  const bool walk_all = MODE == kUpMayWalk && own_list && p.walk_all &&
                        (long long)n_listed * 100 >= (long long)p.R * kWalkAllPercent;
  if (walk_all) n_rows = p.R;
  const int tile_rows = tile_rows_for(n_rows, gridDim.x, p.equal_max);
  const int n_tiles = (n_rows + tile_rows - 1) / tile_rows;
  // Calls put(list position, row) for the rows of the gate tiles of this warp's lanes with `mine`: a lane a row, 32 at a time.  (A
  // thread that went through the set bits of its own word took a microsecond for them.)
  auto each_row = [&](bool mine, auto&& put) {
    unsigned todo = __ballot_sync(0xffffffffu, mine);
    while (todo) {
      const int src = __ffs(todo) - 1;
      todo &= todo - 1;
      int pos = __shfl_sync(0xffffffffu, first_pos, src), j = (tid - lane + src) * p.gate_tile_rows + lane;
#pragma unroll
      for (int i = 0; i < 4; ++i, j += p.gate_rows_per_word) {
        const uint32_t b = __shfl_sync(0xffffffffu, bits[i], src);
        if (b >> lane & 1) put(pos + __popc(b & ((1u << lane) - 1u)), j);
        pos += __popc(b);
      }
    }
  };
  if (own_list && walk_all) {
    // publish the list only: a tile's part is written out by CTA tile mod grid
    each_row(fired_here && tid % (int)gridDim.x == (int)blockIdx.x, [&](int li, int j) { p.idx_out[li] = j; });
    if (blockIdx.x == 0 && tid == 0) {
      *p.count_out = n_listed;
      *p.walk_all = 1;
    }
  } else if (own_list) {
    if (blockIdx.x == 0 && tid == 0 && p.walk_all) *p.walk_all = 0;
    // keep the rows of this CTA's tiles in shared memory and publish them (and the length) for the
    // down projection and the caller: every list position belongs to exactly one CTA's tile
    int m = 0;
    for (int tile = blockIdx.x; tile < n_tiles; tile += gridDim.x, ++m) {
      const int lo = tile * tile_rows, hi = lo + tile_rows;
      each_row(fired_here && first_pos < hi && first_pos + fired_here > lo, [&](int li, int j) {
        if (li >= lo && li < hi) {
          rows_sm[m * kTileRows + li - lo] = j;
          p.idx_out[li] = j;
        }
      });
    }
    if (blockIdx.x == 0 && tid == 0) *p.count_out = n_rows;
  }
  // Stage geometry.  Tiles of up to 64 rows are multiplied with M = 64 (accumulator row i then sits in TMEM lane
  // 32 * (i / 16) + i % 16), taller ones with M = 128 (row i in lane i).  A stage holds `atoms` successive K
  // blocks of the tile -- short tiles take several, so that a stage stays near 16 KB and the bytes in flight do
  // not shrink with the tile -- followed by the token rows of the same K blocks.  Block a sits tile_rows * 128
  // bytes after block a - 1; its MMA reads M rows from its start, i.e. on into the following blocks and the
  // token rows of the same stage (rows that are ignored); the stage is sized so that it never reads past it.
  const bool m64 = !PAIR && tile_rows <= 64;
  const int mrows = m64 ? 64 : kTileRows;
  int atoms = kTileRows / tile_rows;
  const int atoms_cap = npad <= 16 ? 4 : npad <= 32 ? 2 : 1;  // at most 8 KB of token rows per stage
  atoms = atoms > atoms_cap ? atoms_cap : atoms;
  const int a_block_bytes = tile_rows * 128, b_cols = PAIR ? npad / 2 : npad, b_block_bytes = b_cols * 128;
  // bytes of the bf16 weight blocks of a stage, including what the last block's MMA reads past its rows
  const int a_bytes = (max(atoms * a_block_bytes, (atoms - 1) * a_block_bytes + mrows * 128) + 1023) & ~1023;
  const int raw_block_bytes = tile_rows * kRawRow;
  // bf16 rows: a slot holds the weight blocks, then the token rows.  Quantised rows: the ring slots hold what the
  // copies bring (token rows, then the codes), and the expanded bf16 blocks have a short ring of their own (stage
  // `it` uses slot it mod 4 of it): the codes in flight, not the expanded blocks, are what has to cover the memory
  // latency.
  const int b_off = kExp ? 0 : atoms * a_block_bytes;           // token rows within a ring slot
  const int w_off = kExp ? atoms * b_block_bytes : 0;           // weights (as copied) within a ring slot
  int stage_bytes = kExp ? atoms * (b_block_bytes + raw_block_bytes) : max(atoms * (a_block_bytes + b_block_bytes), a_bytes);
  stage_bytes = (stage_bytes + 1023) & ~1023;
  const uint32_t ring0 = stage0 + (kExp ? kExpandSlots * a_bytes : 0);
  int S = (p.ring_bytes - (kExp ? kExpandSlots * a_bytes : 0)) / stage_bytes;
  S = S > (kExp ? kMaxStages : kMaxStagesBf16) ? (kExp ? kMaxStages : kMaxStagesBf16) : S;
  // four issuers when the ring divides evenly among them, otherwise two (slot mod issuers = owner)
  int issuers = (S >= 8 && S % 4 == 0) ? 4 : kExp && S >= 4 ? 4 : 2;
  S &= (kExp && S >= 4) ? ~3 : ~1;
  issuers = issuers > max_acc ? max_acc : issuers;
  if (EX) {
    issuers = exact_issuers(npad);
    S &= ~3;
  }
  const int kstages = (kblocks + atoms - 1) / atoms;
  // accumulator row that this thread's TMEM lane holds (-1: none); the same for every warp of a lane quarter
  const int row_thr = m64 ? (lane < 16 ? (warp & 3) * 16 + lane : -1) : (warp & 3) * 32 + lane;
  // The MMA issuers take the stages of their ring slots (slot mod issuers) into accumulators of their own
  // (npad TMEM columns each); the epilogue adds them.  A tile with at least as many stages as issuers
  // gives each issuer a stage; shorter tiles use fewer issuers.
  const int nacc = kstages >= issuers ? issuers : kstages >= 2 ? 2 : 1;
  if (tid == 0) {
    mbar_init(acc_full, nacc);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  tc_fence_before();
  if constexpr (PAIR) cluster_sync();  // the other CTA's barriers are initialised too
  else __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;

  // Epilogue of one tile for the token-column groups c0 = 8 * part, 8 * (part + nparts), ...: waits for the
  // tile's accumulators, then (gate) adds the fixed-matrix term and the bias, applies the activation and
  // stores the gate values, reporting whether any token fired; (union rows) scales by the gate values
  // and stores HmT.  Returns false if the wait was abandoned.
  const bool share_last = !EX && npad >= 32;  // four or more column groups: worth spreading over all warps
  // `shared`: all twelve warps take part.  Only the epilogue warps have followed the accumulator barrier through
  // every earlier tile (a warp that joins for the last tile could find it still in an earlier phase, which a parity
  // wait cannot tell from "complete"), so they wait for it and the others meet them at a named barrier.
  auto epilogue = [&](int tile, int tcount, int part, int nparts, bool shared, bool& fired) -> bool {
    const int row_in_tile = row_thr;
    const uint32_t taddr = tmem_base + ((uint32_t)((warp & 3) * 32) << 16);
    const int B = p.B;
    const int li = tile * tile_rows + row_in_tile;
    const bool row_ok = row_in_tile >= 0 && row_in_tile < tile_rows && li < n_rows;
    int j = !row_ok ? 0 : (own_list && !walk_all) ? rows_sm[tcount * kTileRows + row_in_tile] : p.idx ? p.idx[li] : li;
    if (!SFFN_IN_BOUNDS(j >= 0 && j < p.R, p.status, 40)) j = 0;
    // everything that does not depend on the accumulator is fetched before the wait
    if (MODE == kGate) pdl_wait();  // before the first read of a buffer an earlier kernel may write, and the first store
    float bias = 0.f, sg = 1.f;
    const float sc = ((kQ && row_ok && p.w_scale) ? p.w_scale[j] : 1.f) * (kI4 ? 0.0625f : 1.f);  // scale of the weight row
    const float osc = (kQ && UP && row_ok && p.out_scale) ? p.out_scale[j] : 1.f;  // scale of the down row, folded into Hm
    int gi = -1;
    if (!UP) {
      bias = (row_ok && p.b_g) ? p.b_g[j] : 0.f;
      gi = (row_ok && p.g_idx) ? p.g_idx[j] : -1;
      sg = (row_ok && p.g_sign && p.g_sign[j] < 0) ? -1.f : 1.f;
    }
    // What a step of the loops below (kStep tokens) needs of each token beside its sums: gate value (union rows) or fixed-matrix
    // entry (gate), and the scale of its limbs.  Two steps are always under way: with the loads where they are used a step waited
    // for each of them in turn.
    constexpr int kStep = kNat ? 4 : 8;
    const __nv_bfloat16* xg = static_cast<const __nv_bfloat16*>(p.xtok) + (gi >= 0 ? gi : 0);
    struct Pre { float e[kStep], ts[kNat ? kStep : 1]; };
    auto fetch = [&](int b0) -> Pre {
      Pre w;
#pragma unroll
      for (int q = 0; q < kStep; ++q) {
        const int b = b0 + q;
        if (UP) w.e[q] = ld_f32_if(p.a + (size_t)b * p.a_stride + j, row_ok && b < B);
        else w.e[q] = ld_bf16_if(xg + (size_t)b * p.xtok_stride, gi >= 0 && b < B);
        if (kNat) w.ts[q] = ld_f32_if(p.tok_scale + b, b < B);
      }
      return w;
    };
    const int b_first = kStep * part, b_step = kStep * nparts;
    Pre now = fetch(b_first), next = fetch(b_first + b_step);
    int okw = 1;
    if (!shared || (warp >= 4 && warp < 8)) {
      if (lane == 0) okw = mbar_wait(acc_full, tcount & 1, abort_flag, p.status, p.wait_cycles) ? 1 : 0;
      okw = __shfl_sync(0xffffffffu, okw, 0);
    }
    if (shared) {
      tc_fence_before();
      named_bar_sync(3, kThreadsRows);  // reached by all twelve warps whatever happened before
      if (*abort_flag) okw = 0;
    }
    if (!okw) return false;
    tc_fence_after();
    if constexpr (kNat) {
      // int32 accumulators, four columns per token (its limbs): value = token scale * row scale * their sum
      if (kSplits && p.k_splits > 1) {  // a run of K: added to the integer sums of the others, in whatever order
#pragma unroll 1
        for (int c0 = 8 * part; c0 < npad; c0 += 8 * nparts) {
          int iv[8];
          tmem_ld8_int(taddr + c0, nacc, npad, iv);
          int* sums = reinterpret_cast<int*>(a_out) + (size_t)c0 * p.a_stride + j;  // column c0 is limb c0 mod 4 of token c0 / 4
#pragma unroll
          for (int q = 0; q < 8; ++q)
            if (row_ok && c0 + q < 4 * B) atomicAdd(sums + (size_t)q * p.a_stride, iv[q]);
        }
        return true;
      }
    }
    // Bound by instruction issue: three warps a scheduler, and code that is fetched anew by every launch.  A step's tokens go
    // through straight-line code, accesses predicated and the activation chosen once for all of them: with a branch around each
    // token a step of eight took 1640 cycles (4096 x 14336, 200 tokens, bf16, after the last MMA of the gate / up kernel: 8.6 / 8.0
    // us, now 5.6 / 5.2; int8, 64 tokens: 4.9 / 7.0 -> 2.9 / 2.6; whole calls 129 -> 123, 88.5 -> 80.7).  Steps of 16 and of 4
    // bf16 tokens are slower (whole calls of 4096 x 14336, 24 / 200 tokens, 16 / 8 / 4: 70.1 / 68.0 / 68.7, 134 / 127 / 129).
#pragma unroll 1
    for (int b0 = b_first; b0 < B; b0 += b_step) {
      float v[kStep];
      if constexpr (kNat) {
        int iv[16];
        tmem_ld16_int(taddr + 4 * b0, nacc, npad, iv);
#pragma unroll
        for (int q = 0; q < kStep; ++q) v[q] = now.ts[q] * sc * limb_sum(iv[4 * q], iv[4 * q + 1], iv[4 * q + 2], iv[4 * q + 3]);
      } else {
        tmem_ld8(taddr + b0, nacc, npad, v);
        if (!UP && p.x_cols) {  // LoPA: a token's vector is the sum of two bf16 vectors (columns b and x_cols + b)
          float w[8];
          tmem_ld8(taddr + p.x_cols + b0, nacc, npad, w);
#pragma unroll
          for (int q = 0; q < 8; ++q) v[q] += w[q];
        }
      }
      const Pre w = now;
      now = next;
      next = fetch(b0 + 2 * b_step);
      if (UP) {
        if (kQ && !kNat) {
#pragma unroll
          for (int q = 0; q < kStep; ++q) v[q] *= sc;
        }
        activate<kStep>(p.act_up, v, B - b0, row_ok);
        __nv_bfloat16* hm = static_cast<__nv_bfloat16*>(p.hmT) + (size_t)b0 * p.hm_stride + li;
#pragma unroll
        for (int q = 0; q < kStep; ++q) {
          float h = kQ ? w.e[q] * v[q] * osc : w.e[q] * v[q];
          if (!kNat) h = fired_part(w.e[q], h);
          const bool on = row_ok && b0 + q < B;
          // one bf16 value, or (quantised rows of some widths) two that add up to 16 bits of h
          if (kQ && !kNat && p.h_terms == 2) {
            st_bf16_if(hm + (size_t)q * p.hm_stride, take_bf16(h), on);
            st_bf16_if(hm + (size_t)(p.h_cols + q) * p.hm_stride, __float2bfloat16(h), on);
          } else {
            st_bf16_if(hm + (size_t)q * p.hm_stride, __float2bfloat16(h), on);
          }
        }
      } else {
#pragma unroll
        for (int q = 0; q < kStep; ++q) {
          v[q] = kQ && !kNat ? v[q] * sc + bias : v[q] + bias;
          v[q] = gi >= 0 ? v[q] + sg * w.e[q] : v[q];
          fired |= (b0 + q < B) & (v[q] > 0.f);
        }
        activate<kStep>(p.act, v, B - b0, row_ok);
        float* arow = a_out + (size_t)b0 * p.a_stride + j;
#pragma unroll
        for (int q = 0; q < kStep; ++q) st_f32_if(arow + (size_t)q * p.a_stride, v[q], row_ok && b0 + q < B);
      }
    }
    return true;
  };

  // EX: the same for the token columns of this warp's set, from sums added in registers; stage `it` of the CTA's sequence
  // comes from ring slot it mod S and issuer it mod issuers (S is a multiple of their number).
  constexpr int kHalf = QB ? kExactHalfTerms : kExactHalf;  // quantised rows: LoPA gates only
  auto exact_epilogue = [&](int tile, int tcount, int set, int& it, int& s, bool& fired) -> bool {
    float sum[kHalf], low[kHalf];
#pragma unroll
    for (int c = 0; c < kHalf; ++c) sum[c] = low[c] = 0.f;
    const uint32_t taddr = tmem_base + ((uint32_t)((warp & 3) * 32) << 16);
    const int li = tile * tile_rows + row_thr;
    const bool row_ok = row_thr >= 0 && row_thr < tile_rows && li < n_rows;
    int j = !row_ok ? 0 : own_list ? rows_sm[tcount * kTileRows + row_thr] : p.idx ? p.idx[li] : li;
    if (!SFFN_IN_BOUNDS(j >= 0 && j < p.R, p.status, 40)) j = 0;
    const int terms = p.x_cols ? 3 : 1, cols = p.x_cols ? p.x_cols : npad;
    const int half = ((cols + 1) / 2 + 7) & ~7, c0 = set * half, c1 = set ? cols : half;
    for (int kb = 0; kb < kstages; ++kb, ++it, ++s) {
      if (s == S) s = 0;
      const int m = it & (issuers - 1);
      int ok = 1;
      if (lane == 0) ok = mbar_wait(place_full + 8 * m, (it / issuers) & 1, abort_flag, p.status, p.wait_cycles) ? 1 : 0;
      if (!__shfl_sync(0xffffffffu, ok, 0)) return false;
      if (warp == 4 && lane == 0) {  // the stage's MMAs are done with their operands
        mbar_arrive(empty + 8 * s);
        if (kExp) mbar_arrive(afree + 8 * (it % kExpandSlots));
      }
      tc_fence_after();
      add_stage<kHalf>(taddr + m * place_cols, min(atoms, kblocks - kb * atoms) * kExactPer, npad, c0, c1, terms, p.x_cols, sum, low);
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(place_empty + 8 * m);
    }
    finish_sums<kHalf>(sum, low);
    if (MODE == kGate) pdl_wait();
    const float sc = (kQ && row_ok && p.w_scale) ? p.w_scale[j] : 1.f;
    if (!row_ok) return true;
    const int B = p.B < c1 ? p.B : c1;
    if (UP) {
      const float osc = (kQ && p.out_scale) ? p.out_scale[j] : 1.f;
      __nv_bfloat16* hm = static_cast<__nv_bfloat16*>(p.hmT) + li;
      const size_t term = (size_t)p.h_cols * p.hm_stride;
#pragma unroll
      for (int i = 0; i < kHalf; ++i) {
        const int b = c0 + i;
        if (b < B) {
          const float av = p.a[(size_t)b * p.a_stride + j];
          float h = av * activation(p.act_up, kQ ? sum[i] * sc : sum[i]);
          if (kQ) h *= osc;
          h = fired_part(av, h);
          // 24 bits of h as three bf16 values
          __nv_bfloat16* dst = hm + (size_t)b * p.hm_stride;
          dst[0] = take_bf16(h);
          dst[term] = take_bf16(h);
          dst[2 * term] = __float2bfloat16(h);
        }
      }
    } else {
      const float bias = p.b_g ? p.b_g[j] : 0.f;
      const int gi = p.g_idx ? p.g_idx[j] : -1;
      const float sg = (p.g_sign && p.g_sign[j] < 0) ? -1.f : 1.f;
      const __nv_bfloat16* xg = static_cast<const __nv_bfloat16*>(p.xtok) + (gi >= 0 ? gi : 0);
#pragma unroll
      for (int i = 0; i < kHalf; ++i) {
        const int b = c0 + i;
        if (b < B) {
          float z = kQ ? sum[i] * sc + bias : sum[i] + bias;
          if (gi >= 0) z += sg * __bfloat162float(xg[(size_t)b * p.xtok_stride]);
          fired |= z > 0.f;
          a_out[(size_t)b * p.a_stride + j] = activation(p.act, z);
        }
      }
    }
    return true;
  };

  if (warp < kProducerWarps) {
    // ======================= producers =========================================================
    // Stages are numbered it = 0, 1, ... over this CTA's (tile, K block) sequence and use ring slot
    // it mod S.  A slot always belongs to the same producer warp (slot mod 4) and the same MMA issuer
    // (slot mod 2, S is even): a waiter that owns its slot can never be two barrier phases behind it,
    // which a parity wait could not tell from "ready".  Lane 0 waits for the slot and announces the byte
    // count, then the copies go out: one tiled copy for the tile's consecutive rows (gate), or one
    // gather4 per lane for four listed rows each (union rows); the token block is one more tiled copy.
    const int my_tiles = first < n_tiles ? (n_tiles - 1 - first) / (int)gridDim.x + 1 : 0;
    const int total = my_tiles * kstages;
    auto copy_tile = [&](uint32_t dst, const CUtensorMap* map, int c0, int c1, uint32_t bar) {
      if constexpr (PAIR) tma_tile_2d_pair(dst, map, c0, c1, bar);
      else tma_tile_2d(dst, map, c0, c1, bar);
    };
    auto copy_gather = [&](uint32_t dst, int c0, const int* r, uint32_t bar) {
      if constexpr (PAIR) tma_gather4_pair(dst, &map_w, c0, r[0], r[1], r[2], r[3], bar);
      else tma_gather4(dst, &map_w, c0, r[0], r[1], r[2], r[3], bar);
    };
    // Stages [it0, it1) of this CTA's sequence; with_w / with_x say which of the two operands are copied.  A
    // stage is armed (slot waited for, byte count announced) together with its weight copy.
    auto produce = [&](int it0, int it1, bool with_w, bool with_x) -> bool {
      int s = it0 % S, ph = (it0 / S) & 1, kb = it0 % kstages, tl = it0 / kstages;
      int rows_of = -1;
      int r[4] = {0, 0, 0, 0};
      for (int it = it0; it < it1; ++it, ++s, ++kb) {
        if (s == S) { s = 0; ph ^= 1; }
        if (kb == kstages) { kb = 0; ++tl; }
        if ((s & (kProducerWarps - 1)) != warp) continue;
        const int tile = blockIdx.x + tl * gridDim.x;
        const int na = min(atoms, kblocks - kb * atoms);
        // PAIR: the bytes of both CTAs, whose copies complete on the even one's barrier
        const uint32_t tx_bytes = (PAIR ? 2 : 1) * (kExp ? (uint32_t)(na * (tile_rows * kRawRow + b_cols * 128)) : (uint32_t)(na * (tile_rows + b_cols)) * 128);
        const uint32_t bar = PAIR ? map_rank(full + 8 * s, 0) : full + 8 * s;
        if (UP && !walk_all && tl != rows_of) {
          rows_of = tl;
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            const int li = tile * tile_rows + lane * 4 + q;
            // rows beyond the list or the tile: row 0, ignored later
            r[q] = (li >= n_rows || lane * 4 + q >= tile_rows) ? 0
                   : own_list ? rows_sm[tl * kTileRows + lane * 4 + q] : p.idx ? p.idx[li] : li;
            if (!SFFN_IN_BOUNDS(r[q] >= 0 && r[q] < p.R, p.status, 41)) r[q] = 0;
          }
        }
        if (with_w) {
          int ok = 1;
          if (lane == 0) {
            ok = mbar_wait(empty + 8 * s, ph ^ 1, abort_flag, p.status, p.wait_cycles) ? 1 : 0;
            if (ok && rank == 0) mbar_expect_tx(full + 8 * s, tx_bytes);
          }
          ok = __shfl_sync(0xffffffffu, ok, 0);
          if (!ok) return false;
        }
        const uint32_t abase = ring0 + s * stage_bytes;
        for (int a = 0; a < na; ++a) {
          const int k0 = (kb_first + kb * atoms + a) * kAtomElems;
          // where the weight block lands, the byte column it starts at, and the bytes of one landed row
          const uint32_t wdst = abase + w_off + a * (kExp ? raw_block_bytes : a_block_bytes);
          const int wc0 = kI4 ? k0 / 2 : kExp ? k0 * QB / 8 : k0;
          const int wrow = kExp ? kRawRow : 128;
          if (with_w && !(MODE == kGate && blockIdx.x == 0 && it == p.drop_stage)) {  // test hook: a copy that never comes
            if (UP && !walk_all) {
              if (lane * 4 < tile_rows)
                copy_gather(wdst + lane * 4 * wrow, wc0, r, bar);
            } else if (UP) {
              if (lane == 0) copy_tile(wdst, map_t.get(), wc0, tile * tile_rows, bar);
            } else if (lane == 0) {
              copy_tile(wdst, &map_w, wc0, tile * tile_rows, bar);
            }
          }
          if (with_x && lane == 0) copy_tile(abase + b_off + a * b_block_bytes, &map_x, k0, rank * b_cols, bar);
        }
      }
      return true;
    };
    if (MODE == kGate) {
      // the first ring-full of weight tiles goes out while the predecessor in the stream still runs; the token
      // rows of those stages follow once it has finished
      const int ahead = total < S ? total : S;
      const bool ok = produce(0, ahead, true, false);
      pdl_wait();
      if (ok && produce(0, ahead, false, true)) produce(ahead, total, true, true);
    } else {
      produce(0, total, true, true);
    }
  } else if (kExp && warp >= kExpand0 / 32) {
    // ======================= expanders (quantised rows): codes -> bf16 block of the slot ==========
    // Two pairs of warps; a pair takes the slots of its parity (S is even), in the producers' order, so it meets
    // every phase of its slots and cannot fall two phases behind; while one pair waits the other one converts.
    const int my_tiles = first < n_tiles ? (n_tiles - 1 - first) / (int)gridDim.x + 1 : 0;
    const int total = my_tiles * kstages;
    const int pair = (tid - kExpand0) / (16 * kExpandWarps);
    const int et = (tid - kExpand0) % (16 * kExpandWarps);
    int s = 0, ph = 0, kb = 0;
    for (int it = 0; it < total; ++it, ++s, ++kb) {
      if (s == S) { s = 0; ph ^= 1; }
      if (kb == kstages) kb = 0;
      if ((s & 1) != pair) continue;
      const int t = it % kExpandSlots;
      // the codes have landed, and the MMAs of the stage that used the bf16 slot before are done
      const bool ok = mbar_wait(full + 8 * s, ph, abort_flag, p.status, p.wait_cycles) &&
                      mbar_wait(afree + 8 * t, ((it / kExpandSlots) & 1) ^ 1, abort_flag, p.status, p.wait_cycles);
      if (!__all_sync(0xffffffffu, ok)) break;
      const uint32_t src = ring0 + s * stage_bytes + w_off, dst = stage0 + t * a_bytes;
      const int na = min(atoms, kblocks - kb * atoms);
      for (int a = 0; a < na; ++a)
        if (kI4) expand_block_q4_i8<QB == 3 ? 8 : 1>(src + a * raw_block_bytes, dst + a * a_block_bytes, tile_rows, et, 16 * kExpandWarps);
        else expand_block<(QB == 8 || QB == 4) ? QB : 8>(src + a * raw_block_bytes, dst + a * a_block_bytes, tile_rows, et, 16 * kExpandWarps);
      fence_proxy_async();
      __syncwarp();
      if (lane == 0) mbar_arrive(ready + 8 * t);
    }
  } else if (warp >= 8 && warp < kThreadsRows / 32) {
    // ======================= MMA issuers =======================================================
    const int m = warp - 8;
    if constexpr (EX) {
      if (lane == 0 && m < issuers) {
        const uint32_t idesc = make_idesc(npad, mrows);
        const uint32_t place = tmem_base + m * place_cols;
        const int my_tiles = first < n_tiles ? (n_tiles - 1 - first) / (int)gridDim.x + 1 : 0;
        int s = 0, ph = 0, kb = 0;
        for (int it = 0; it < my_tiles * kstages; ++it, ++s, ++kb) {
          if (s == S) { s = 0; ph ^= 1; }
          if (kb == kstages) kb = 0;
          if ((it & (issuers - 1)) != m) continue;  // another issuer's slot
          const int t = it % kExpandSlots;
          if (kExp ? !mbar_wait(ready + 8 * t, (it / kExpandSlots) & 1, abort_flag, p.status, p.wait_cycles)
                   : !mbar_wait(full + 8 * s, ph, abort_flag, p.status, p.wait_cycles)) break;
          if (!mbar_wait(place_empty + 8 * m, ((it / issuers) & 1) ^ 1, abort_flag, p.status, p.wait_cycles)) break;
          tc_fence_after();
          const uint32_t sbase = ring0 + s * stage_bytes;
          const uint32_t wbase = kExp ? stage0 + t * a_bytes : sbase;
          const int na = min(atoms, kblocks - kb * atoms);
          for (int a = 0; a < na; ++a) {
            const uint64_t adesc = make_desc(wbase + a * a_block_bytes);
            const uint64_t bdesc = make_desc(sbase + b_off + a * b_block_bytes);
#pragma unroll
            for (int k = 0; k < kAtomK / 16; ++k)
              umma(place + (a * kExactPer + k / kExactMmas) * npad, adesc + 2 * k, bdesc + 2 * k, idesc, k % kExactMmas ? 1u : 0u);
          }
          umma_commit(place_full + 8 * m);
        }
      }
    } else if (lane == 0 && m < nacc && rank == 0) {
      const uint32_t idesc = kNat ? make_idesc_i8(npad, PAIR ? 2 * mrows : mrows) : make_idesc(npad, PAIR ? 2 * mrows : mrows);
      auto mma = [&](uint32_t d, uint64_t adesc, uint64_t bdesc, uint32_t accumulate) {
        if constexpr (PAIR && kNat) umma_pair_i8(d, adesc, bdesc, idesc, accumulate);
        else if constexpr (PAIR) umma_pair(d, adesc, bdesc, idesc, accumulate);
        else if constexpr (kNat) umma_i8(d, adesc, bdesc, idesc, accumulate);
        else umma(d, adesc, bdesc, idesc, accumulate);
      };
      auto commit = [&](uint32_t bar) {
        if constexpr (PAIR) umma_commit_pair(bar);
        else umma_commit(bar);
      };
      const uint32_t acc = tmem_base + m * npad;
      int tcount = 0;
      bool ok = true;
      for (int tile = first; ok && tile < n_tiles; tile += gridDim.x, ++tcount) {
        if (!mbar_wait(acc_empty, (tcount & 1) ^ 1, abort_flag, p.status, p.wait_cycles)) break;
        tc_fence_after();
        const int it0 = tcount * kstages;
        int s = it0 % S, ph = (it0 / S) & 1;
        for (int kb = 0; kb < kstages; ++kb, ++s) {
          if (s == S) { s = 0; ph ^= 1; }
          if ((s & (nacc - 1)) != m) continue;   // another issuer's slot
          const int t = (it0 + kb) % kExpandSlots;  // quantised rows: slot of the bf16 ring
          if (kExp ? !mbar_wait(ready + 8 * t, ((it0 + kb) / kExpandSlots) & 1, abort_flag, p.status, p.wait_cycles)
                 : !mbar_wait(full + 8 * s, ph, abort_flag, p.status, p.wait_cycles)) { ok = false; break; }
          tc_fence_after();
          const uint32_t sbase = ring0 + s * stage_bytes;
          const uint32_t wbase = kExp ? stage0 + t * a_bytes : sbase;
          const int na = min(atoms, kblocks - kb * atoms);
          for (int a = 0; a < na; ++a) {
            const uint64_t adesc = make_desc(wbase + a * a_block_bytes);
            const uint64_t bdesc = make_desc(sbase + b_off + a * b_block_bytes);
            mma(acc, adesc, bdesc, (kb >= nacc || a > 0) ? 1u : 0u);
#pragma unroll
            for (int k = 1; k < 4; ++k) mma(acc, adesc + 2 * k, bdesc + 2 * k, 1u);
          }
          commit(empty + 8 * s);   // slot free once these MMAs have read it
          if (kExp) commit(afree + 8 * t);
        }
        if (ok) commit(acc_full);  // this issuer's accumulator is complete
      }
    }
    __syncwarp();
  } else {
    // ======================= epilogue warps (wide batches: every tile but the CTA's last) =========
    const int set = EX && warp >= kThreadsRows / 32 ? 1 : 0;
    if (UP && blockIdx.x == 0 && set == 0) {
      // the down projection walks the list in blocks of 64 rows: entries past its end must read as zero
      __nv_bfloat16* hm = static_cast<__nv_bfloat16*>(p.hmT);
      const int end = (n_rows + 63) & ~63;
      for (int li = n_rows + (warp - 4) * 32 + lane; li < end; li += 128)
        for (int b = 0; b < p.B; ++b) {
          hm[(size_t)b * p.hm_stride + li] = __float2bfloat16(0.f);
          if (EX || (kQ && p.h_terms == 2)) hm[(size_t)(p.h_cols + b) * p.hm_stride + li] = __float2bfloat16(0.f);
          if (EX) hm[(size_t)(2 * p.h_cols + b) * p.hm_stride + li] = __float2bfloat16(0.f);
        }
    }
    int tcount = 0, it = 0, s = 0;
    int tile = blockIdx.x;  // PAIR: all of the pair's tiles but its last one here, whose shared epilogue both CTAs go through
    // which rows of the tile fired, as the up kernel or the compaction reads it
    auto publish = [&](bool fired) {
      const int li = tile * tile_rows + row_thr;
      const bool valid = row_thr >= 0 && row_thr < tile_rows && li < n_rows;
      if (p.flag && valid) p.flag[li] = fired ? 1 : 0;
      if (p.words_out) {
        const unsigned m = __ballot_sync(0xffffffffu, fired && valid);
        if (lane == 0 && tile < n_tiles) p.words_out[4 * tile + (warp & 3)] = m;
      }
    };
    for (; tile - rank + (share_last ? (int)gridDim.x : 0) < n_tiles; tile += gridDim.x, ++tcount) {
      bool fired = false;
      if constexpr (EX) {
        const bool done = exact_epilogue(tile, tcount, set, it, s, fired);
        if (UP) {
          if (!done) break;
          continue;
        }
        // the two sets of warps hold the flags of half of the tokens each; both leave together
        uint8_t* fired_sm = reinterpret_cast<uint8_t*>(scan_wt) + (tcount & 1) * 2 * kTileRows;  // the scan scratch is free here
        const int me = (warp & 3) * 32 + lane;
        fired_sm[set * kTileRows + me] = fired ? 1 : 0;
        if (named_bar_any(2, 256, !done)) break;
        if (set) continue;
        fired = (fired_sm[me] | fired_sm[kTileRows + me]) != 0;
      } else {
        if (!epilogue(tile, tcount, 0, 1, false, fired)) break;
      }
      if (!UP) publish(fired);
      if (EX) continue;
      tc_fence_before();
      if constexpr (PAIR) mbar_arrive_cluster(map_rank(acc_empty, 0));
      else mbar_arrive(acc_empty);
    }
    // after a wait that ran out: nothing fired in the tiles that are left (the masks there are an earlier call's, or
    // the bytes of another route, whose bits need not stand for rows at all)
    if (!UP && set == 0)
      for (; tile - rank + (share_last ? (int)gridDim.x : 0) < n_tiles; tile += gridDim.x) {
        pdl_wait();
        publish(false);
      }
  }

  // ---- the CTA's last tile (wide batches): by now the producer and issuer warps have nothing left to do, so
  // all twelve warps share its epilogue.  A warp reads the TMEM lanes of its quarter (warp mod 4); the three warps of
  // a quarter take every third group of eight token columns.
  if (share_last && first < n_tiles && warp < kThreadsRows / 32) {
    const int my_tiles = (n_tiles - 1 - first) / (int)gridDim.x + 1;
    const int last_tile = blockIdx.x + (my_tiles - 1) * gridDim.x;
    const int part = warp >= 8 ? 2 : warp >= 4 ? 0 : 1;
    bool fired = false;
    const bool done = epilogue(last_tile, my_tiles - 1, part, 3, true, fired);
    if (!UP && (p.flag || p.words_out)) {
      uint8_t* fired_sm = reinterpret_cast<uint8_t*>(scan_wt);  // [3][128], the scan scratch is free here
      const int row_in_tile = row_thr;
      const int me = (warp & 3) * 32 + lane;  // this thread's entry: the same in all three parts
      fired_sm[part * kTileRows + me] = fired ? 1 : 0;
      named_bar_sync(2, kThreadsRows);  // reached by every thread of a CTA that owns a tile, whatever happened
      const int li = last_tile * tile_rows + row_in_tile;
      if (part == 0) {  // warps 4-7, all lanes
        const bool valid = done && row_in_tile >= 0 && row_in_tile < tile_rows && li < n_rows;
        const bool any = (fired_sm[me] | fired_sm[kTileRows + me] | fired_sm[2 * kTileRows + me]) != 0;
        if (p.flag && valid) p.flag[li] = any ? 1 : 0;
        if (p.words_out) {
          const unsigned m = __ballot_sync(0xffffffffu, any && valid);
          if (lane == 0 && last_tile < n_tiles) p.words_out[4 * last_tile + (warp & 3)] = m;
        }
      }
    }
  }

  // ---- teardown: everybody meets, then the allocating warp frees the TMEM columns ------------------
  // (after a wait that ran out, copies and MMAs may still be in flight: they end within microseconds, and shared
  // memory and TMEM are only given back after that)
  if (*abort_flag)
    for (int i = 0; i < 50; ++i) __nanosleep(1000);
  tc_fence_before();
  // (PAIR: nor is there shared memory left behind that the even CTA's MMAs, or its commits, reach for)
  if constexpr (PAIR) cluster_sync();
  else __syncthreads();
  if (PAIR && warp == 8) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(tmem_cols) : "memory");
  } else if (warp == 8) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(tmem_cols) : "memory");
  }
}

// ------------------------------------------------------------------------------------------------
// Down projection over the union list (Sec. 5.4): y[b][d] = sum over the listed rows u of Hm[b][u] * W_down[idx[u]][d].
// One CTA owns 128 output columns d (TMEM lanes) and one split of the list, a cluster (if any) all splits of those columns;
// the contraction runs over list rows, so the gathered W_down rows are the MN-major A operand (each
// gathered row delivers 64 contiguous d per swizzle row) and HmT[b][u] is the K-major B operand.
// Same pipeline as above: 4 producer warps (gather4 per lane: 2 column halves x 16 row quads = one 64-row
// stage), 2 MMA issuers with their own accumulators, 4 epilogue warps, which the producers join; two CTAs share an SM.
// Threads, rounded up to whole warps for each scheduler: registers are handed out by scheduler, and two CTAs of 14 warps with 72
// registers a thread, which fit an SM's file, do not fit those of the first two (int4 rows ran in two waves of CTAs).
constexpr int down_bound(int qb, bool exact) { return ((exact ? 512 : kThreads) + (qb ? 32 * kExpandWarps : 0) + 127) / 128 * 128; }
// CL: calls whose splits may be clusters.  Exact sums of codes, whose kernel fills its registers and spills a few, have another one without
// that code for the calls that have none (LoPA gate, 7296 x 21888, 39 / 64 tokens, with / without: int8 495 / 864 -> 487 / 851 us, int4 488 /
// 851 -> 480 / 837; bf16 rows, which spill nothing, are 2 % slower so: 746 -> 756).
template <int QB, bool EX = false, bool TWO = false, bool CL = true>
__global__ void __launch_bounds__(down_bound(QB, EX), EX ? 1 : 2) umma_down_kernel(const UmmaDownParams p,
                                                                  const __grid_constant__ CUtensorMap map_wg,
                                                                  const __grid_constant__ CUtensorMap map_wt,
                                                                  const __grid_constant__ CUtensorMap map_hm) {
  extern __shared__ __align__(1024) unsigned char smem_raw[];
  const int npad = p.npad;
  constexpr int kRawBytes = QB * kTileRows * kAtomK / 8;  // quantised rows: the codes of a stage's 64 rows x 128 columns
  // Quantised rows.  One ring: a slot holds the expanded block, h, then the codes.  TWO: it holds what the copies bring (h, then
  // the codes); the expanded blocks have a short ring of their own in front of it (stage kb uses block kb mod E), as in the rows
  // kernels.  That is for the slots that with room for both are two or four (see launch_umma_down; whole calls, int8, 4096 x
  // 14336, 24 / 64 tokens, one ring / two: 70.6 / 97.5 -> 62.4 / 88.7 us; 8192 x 18000, 24 tokens: 142 -> 116).
  constexpr bool kTwo = TWO;
  static_assert(!TWO || (QB != 0 && !EX), "two rings: codes, plain sums");
  const int E = p.expand, expand_bytes = kTwo ? E * kAAtomBytes : 0;
  const int b_off = kTwo ? 0 : kAAtomBytes;               // h within a slot
  const int raw_off = b_off + npad * 128;
  const int stage_bytes = raw_off + kRawBytes;
  const int S = p.stages;
  unsigned char* smem = reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem + p.ring_bytes);  // (the rings, or as much as the sums of the tokens take)
  const uint32_t expand0 = smem_u32(smem), stage0 = expand0 + expand_bytes;
  const uint32_t full = smem_u32(bars), empty = smem_u32(bars + S);
  const uint32_t acc_full = smem_u32(bars + 2 * S);
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + 2 * S + 2);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
  const uint32_t ready = smem_u32(bars + 2 * S + 4);  // expanded block written (kTwo: one per block, else one per slot) ...
  const uint32_t afree = ready + 8 * kDownExpand;     // ... kTwo: and read by its MMAs

  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int d_tiles = p.D / kTileRows;
  const bool clustered = CL && p.y != nullptr;  // the splits of a tile are one cluster
  const int dt = clustered ? blockIdx.x / p.splits : blockIdx.x % d_tiles, sp = clustered ? blockIdx.x % p.splits : blockIdx.x / d_tiles;
  const int d0 = dt * kTileRows;

  pdl_launch_dependents();
  // EX: see exact sums above; S is a multiple of the issuers, warps 12-15 are the second epilogue set
  const int place_cols = kExactPer * npad, issuers = exact_issuers(npad);
  const uint32_t place_full = ready + 8 * S, place_empty = place_full + 8 * kMaxIssuers;
  constexpr int kExpand0 = EX ? 512 : kThreads;  // first expander thread
  const uint32_t tmem_cols = tmem_cols_for(EX ? issuers * place_cols : 2 * npad);
  if (tid == 0) {
    for (int s = 0; s < S; ++s) {
      mbar_init(full + 8 * s, 1);
      mbar_init(empty + 8 * s, 1);
      if (QB && !kTwo) mbar_init(ready + 8 * s, kExpandWarps / 2);
    }
    if (kTwo)
      for (int e = 0; e < E; ++e) {
        mbar_init(ready + 8 * e, kExpandWarps / 2);
        mbar_init(afree + 8 * e, 1);
      }
    if (EX)
      for (int q = 0; q < kMaxIssuers; ++q) {
        mbar_init(place_full + 8 * q, 1);
        mbar_init(place_empty + 8 * q, 8);
      }
    *abort_flag = 0;
    asm volatile("prefetch.tensormap [%0];" ::"l"(&map_wg) : "memory");
    asm volatile("prefetch.tensormap [%0];" ::"l"(&map_wt) : "memory");
    asm volatile("prefetch.tensormap [%0];" ::"l"(&map_hm) : "memory");
  }
  if (warp == 8) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)),
                 "r"(tmem_cols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  pdl_wait();

  // both words are fetched at once (one round trip), then combined
  const int listed = p.count ? __ldcg(p.count) : p.R;
  const int walk_word = p.walk_all ? __ldcg(p.walk_all) : 0;
  const bool walk_all = p.idx == nullptr || walk_word != 0;  // every row, not the list
  const int n_rows = walk_all ? p.R : listed;
  // the split's share of the list, in blocks of 64 rows
  const int total_blocks = (n_rows + kAtomK - 1) / kAtomK;
  const int per_split = (total_blocks + p.splits - 1) / p.splits;
  const int kb0 = sp * per_split;
  const int kblocks = min(total_blocks, kb0 + per_split) - kb0;  // <= 0: nothing to add, the partial is zero
  const int nacc = kblocks >= 2 ? 2 : 1;
  if (tid == 0) {
    mbar_init(acc_full, nacc);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;

  if (warp < kProducerWarps) {
    // ======================= producers (slot s belongs to warp s mod 4) =========================
    const int terms = QB || EX ? p.terms : 1;
    const uint32_t tx_bytes = (uint32_t)((QB ? kRawBytes : kAAtomBytes) + terms * p.cols * 128);
    const int half = lane >> 4, quad = lane & 15;
    constexpr int kHalfBytes = QB ? kRawBytes / 2 : kAAtomBytes / 2;  // landed bytes of 64 rows x 64 columns
    constexpr int kColDiv = QB == 4 ? 2 : 1;                          // codes per byte
    int s = 0, ph = 0;
    for (int kb = 0; kb < kblocks; ++kb, ++s) {
      if (s == S) { s = 0; ph ^= 1; }
      if ((s & (kProducerWarps - 1)) != warp) continue;
      const int u0 = (kb0 + kb) * kAtomK;
      int r[4] = {0, 0, 0, 0};
      if (!walk_all) {
        // four list entries of this lane (the list buffer is readable past its length; entries there are
        // replaced by row 0, whose products vanish against the zeroed tail of HmT)
        const int u = u0 + quad * 4;
        const int4 v = *reinterpret_cast<const int4*>(p.idx + u);
        r[0] = u + 0 < n_rows ? v.x : 0;
        r[1] = u + 1 < n_rows ? v.y : 0;
        r[2] = u + 2 < n_rows ? v.z : 0;
        r[3] = u + 3 < n_rows ? v.w : 0;
#pragma unroll
        for (int q = 0; q < 4; ++q)
          if (!SFFN_IN_BOUNDS(r[q] >= 0 && r[q] < p.R, p.status, 42)) r[q] = 0;
      }
      int ok = 1;
      if (lane == 0) {
        ok = mbar_wait(empty + 8 * s, ph ^ 1, abort_flag, p.status, p.wait_cycles) ? 1 : 0;
        if (ok) mbar_expect_tx(full + 8 * s, tx_bytes);
      }
      ok = __shfl_sync(0xffffffffu, ok, 0);
      if (!ok) break;
      const uint32_t abase = stage0 + s * stage_bytes;
      const uint32_t wdst = QB ? abase + raw_off : abase;
      if (!walk_all) {
        tma_gather4(wdst + half * kHalfBytes + quad * (kHalfBytes / 16), &map_wg, (d0 + half * kAtomK) / kColDiv, r[0], r[1],
                    r[2], r[3], full + 8 * s);
      } else if (lane < 2) {
        // every row: 64 consecutive rows per column half; rows past the matrix read as zero
        tma_tile_2d(wdst + lane * kHalfBytes, &map_wt, (d0 + lane * kAtomK) / kColDiv, u0, full + 8 * s);
      }
      if (lane < terms)
        tma_tile_2d(abase + b_off + lane * p.cols * 128, &map_hm, u0, lane * p.h_cols + p.tok0, full + 8 * s);
    }
  } else if (QB && warp >= kExpand0 / 32) {
    // ======================= expanders (quantised rows): the stage's codes -> its two bf16 blocks =
    // two pairs of warps, each with the slots of its parity (S is even)
    const int pair = (tid - kExpand0) / (16 * kExpandWarps);
    const int et = (tid - kExpand0) % (16 * kExpandWarps);
    int s = 0, ph = 0;
    for (int kb = 0; kb < kblocks; ++kb, ++s) {
      if (s == S) { s = 0; ph ^= 1; }
      if ((s & 1) != pair) continue;
      const int e = kb & (E - 1);  // (of the parity of s, as S is even)
      const bool ok = mbar_wait(full + 8 * s, ph, abort_flag, p.status, p.wait_cycles) &&
                      (!kTwo || mbar_wait(afree + 8 * e, (kb & E) ? 0u : 1u, abort_flag, p.status, p.wait_cycles));
      if (!__all_sync(0xffffffffu, ok)) break;
      const uint32_t raw = stage0 + s * stage_bytes + raw_off;
      const uint32_t dst = kTwo ? expand0 + e * kAAtomBytes : stage0 + s * stage_bytes;
      if constexpr (QB == 4) {
        expand_block_q4_mn(raw, dst, et);
        expand_block_q4_mn(raw + kRawBytes / 2, dst + kAAtomBytes / 2, et);
      } else {
        static_assert(kAtomK == 16 * kExpandWarps, "four rows a thread");
        expand_block<8, true>(raw, dst, kAtomK, et, 16 * kExpandWarps);
        expand_block<8, true>(raw + kRawBytes / 2, dst + kAAtomBytes / 2, kAtomK, et, 16 * kExpandWarps);
      }
      fence_proxy_async();
      __syncwarp();
      if (lane == 0) mbar_arrive(ready + 8 * (kTwo ? e : s));
    }
  } else if (warp >= 8 && warp < 12) {
    // ======================= MMA issuers (slot s belongs to issuer s mod 2) =====================
    const int m = warp - 8;
    if constexpr (EX) {
      if (lane == 0 && m < issuers) {
        const uint32_t idesc = make_idesc(npad) | (1u << 15);  // A is MN-major
        const uint32_t place = tmem_base + m * place_cols;
        int s = 0, ph = 0;
        for (int kb = 0; kb < kblocks; ++kb, ++s) {
          if (s == S) { s = 0; ph ^= 1; }
          if ((kb & (issuers - 1)) != m) continue;
          if (!mbar_wait((QB ? ready : full) + 8 * s, ph, abort_flag, p.status, p.wait_cycles)) break;
          if (!mbar_wait(place_empty + 8 * m, ((kb / issuers) & 1) ^ 1, abort_flag, p.status, p.wait_cycles)) break;
          tc_fence_after();
          const uint32_t sbase = stage0 + s * stage_bytes;
          const uint64_t bdesc = make_desc(sbase + kAAtomBytes);
#pragma unroll
          for (int k = 0; k < kAtomK / 16; ++k)
            umma(place + k / kExactMmas * npad, make_desc_mn(sbase + k * 2048, 8192, 1024), bdesc + 2 * k, idesc, k % kExactMmas ? 1u : 0u);
          umma_commit(place_full + 8 * m);
        }
      }
    } else if (lane == 0 && m < nacc) {
      const uint32_t idesc = make_idesc(npad) | (1u << 15);  // A is MN-major
      const uint32_t acc = tmem_base + m * npad;
      int s = 0, ph = 0;
      bool ok = true;
      for (int kb = 0; kb < kblocks; ++kb, ++s) {
        if (s == S) { s = 0; ph ^= 1; }
        if (nacc == 2 && (s & 1) != m) continue;
        const int e = kb & (E - 1);
        if (!(kTwo ? mbar_wait(ready + 8 * e, (kb & E) ? 1u : 0u, abort_flag, p.status, p.wait_cycles)
                   : mbar_wait((QB ? ready : full) + 8 * s, ph, abort_flag, p.status, p.wait_cycles))) { ok = false; break; }
        tc_fence_after();
        const uint32_t sbase = stage0 + s * stage_bytes;
        const uint32_t abase = kTwo ? expand0 + e * kAAtomBytes : sbase;
        const uint64_t bdesc = make_desc(sbase + b_off);
#pragma unroll
        for (int k = 0; k < kAtomK / 16; ++k)  // 16 list rows = two groups of eight swizzle rows
          umma(acc, make_desc_mn(abase + k * 2048, 8192, 1024), bdesc + 2 * k, idesc, (kb >= nacc || k > 0) ? 1u : 0u);
        umma_commit(empty + 8 * s);
        if (kTwo) umma_commit(afree + 8 * e);
      }
      if (ok && kblocks > 0) umma_commit(acc_full);
    }
    __syncwarp();
  } else {
    // (below: every warp that has nothing left to do takes part in the epilogue)
  }

  // ======================= epilogue: lane = output column d, TMEM columns = tokens ================
  // Clustered: the split's sums go to shared memory, [token][128 columns] over the ring, which nothing is copied into or multiplied
  // from any more; then each CTA of the cluster adds a share of the tokens up over all splits, in their order.  Else they go to the
  // partials, which a kernel adds up in the same order.
  float* sums = reinterpret_cast<float*>(smem);
  const int B = p.B;
  {
    const int ew = warp & 3;
    const int col = QB == 4 ? column_of_row(ew * 32 + lane) : ew * 32 + lane;
    float* mine = clustered ? sums + col : p.partial + (size_t)sp * B * p.D + d0 + col;
    const size_t pitch = clustered ? kTileRows : p.D;
    const uint32_t taddr = tmem_base + ((uint32_t)(ew * 32) << 16);
    if constexpr (EX) {
      if ((warp >= 4 && warp < 8) || (warp >= 12 && warp < 16)) {
        constexpr int kHalf = QB ? kExactHalfTerms : kExactHalf;
        const int set = warp >= 12 ? 1 : 0;
        float sum[kHalf], low[kHalf];
#pragma unroll
        for (int c = 0; c < kHalf; ++c) sum[c] = low[c] = 0.f;
        const int half = ((p.cols + 1) / 2 + 7) & ~7, c0 = set * half, c1 = set ? p.cols : half;
        int ok = 1, s = 0;
        for (int kb = 0; kb < kblocks; ++kb, ++s) {
          if (s == S) s = 0;
          const int m = kb & (issuers - 1);
          if (lane == 0) ok = mbar_wait(place_full + 8 * m, (kb / issuers) & 1, abort_flag, p.status, p.wait_cycles) ? 1 : 0;
          ok = __shfl_sync(0xffffffffu, ok, 0);
          if (!ok) break;
          if (warp == 4 && lane == 0) mbar_arrive(empty + 8 * s);  // the stage's MMAs are done with their operands
          tc_fence_after();
          add_stage<kHalf>(taddr + m * place_cols, kExactPer, npad, c0, c1, p.terms, p.cols, sum, low);
          tc_fence_before();
          __syncwarp();
          if (lane == 0) mbar_arrive(place_empty + 8 * m);
        }
        finish_sums<kHalf>(sum, low);
#pragma unroll
        for (int i = 0; i < kHalf; ++i)
          if (c0 + i < c1 && c0 + i < B) mine[(c0 + i) * pitch] = sum[i];
      }
    } else if (warp < 8) {
      // two warps for each quarter of the lanes, on alternate groups of eight tokens (there is one phase of this barrier, so any
      // warp may wait for it)
      int okw = 1;
      if (kblocks > 0) {
        if (lane == 0) okw = mbar_wait(acc_full, 0, abort_flag, p.status, p.wait_cycles) ? 1 : 0;
        okw = __shfl_sync(0xffffffffu, okw, 0);
      }
      tc_fence_after();
      const bool some = okw && kblocks > 0;
#pragma unroll 1
      for (int c0 = warp < 4 ? 8 : 0; c0 < B; c0 += 16) {
        float v[8];
#pragma unroll
        for (int q = 0; q < 8; ++q) v[q] = 0.f;
        if (some) {
          tmem_ld8(taddr + c0, nacc, npad, v);
          if (QB && p.terms == 2) {
            float w[8];
            tmem_ld8(taddr + p.cols + c0, nacc, npad, w);
#pragma unroll
            for (int q = 0; q < 8; ++q) v[q] += w[q];
          }
        }
#pragma unroll
        for (int q = 0; q < 8; ++q)
          if (c0 + q < B) mine[(c0 + q) * pitch] = v[q];
      }
    }
  }

  if (*abort_flag)
    for (int i = 0; i < 50; ++i) __nanosleep(1000);
  tc_fence_before();
  // The TMEM goes back before this CTA waits for the others of its cluster.  A CTA whose allocation waits for columns waits without a
  // limit, for a CTA of another stream's call that holds them on its SM; were that one waiting for its own cluster meanwhile, whose
  // other CTA may be the one that cannot allocate on the next SM, neither would ever go on.
  if (clustered) cluster_arrive();
  __syncthreads();
  if (warp == 8) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(tmem_cols) : "memory");
  }
  if (!clustered) return;
  cluster_wait();
  // a warp takes a token at a time, a lane four columns of it
  const int n_warps = blockDim.x >> 5;
  const uint32_t at = smem_u32(sums) + lane * 16;
  for (int b = sp * n_warps + warp; b < B; b += p.splits * n_warps) {
    float4 t = make_float4(0.f, 0.f, 0.f, 0.f);
    for (int r0 = 0; r0 < p.splits; r0 += 4) {
      float4 v[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        v[i] = make_float4(0.f, 0.f, 0.f, 0.f);
        if (r0 + i < p.splits)
          asm volatile("ld.shared::cluster.v4.f32 {%0,%1,%2,%3}, [%4];" : "=f"(v[i].x), "=f"(v[i].y), "=f"(v[i].z), "=f"(v[i].w)
                       : "r"(map_rank(at + b * (kTileRows * 4), r0 + i)) : "memory");
      }
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        t.x += v[i].x;
        t.y += v[i].y;
        t.z += v[i].z;
        t.w += v[i].w;
      }
    }
    *reinterpret_cast<float4*>(p.y + (size_t)b * p.D + d0 + 4 * lane) = t;
  }
  cluster_sync();  // no CTA leaves while another reads its sums
}

// The entries of v for the norm kernels below: the sum of `runs` fp32 values, `step` apart, or the four limbs' integer sums over
// all runs of K (see umma_k_splits), from which v gets the bits that it has without runs.
struct SumVec {
  float* v;
  int stride, runs;
  size_t step;
  __device__ __forceinline__ void token(int b) { v += (size_t)b * stride; }
  __device__ __forceinline__ float entry(int k) const {
    float e = v[k];
#pragma unroll 8
    for (int i = 1; i < runs; ++i) e += v[i * step + k];
    return e;
  }
  __device__ __forceinline__ float& home(int k) const { return v[k]; }
};
struct LimbSumsVec {
  int* v;
  int stride;
  const float *row_scale, *tok_scale;
  float code_scale, tok;
  __device__ __forceinline__ void token(int b) { v += (size_t)4 * b * stride, tok = tok_scale[b]; }
  __device__ __forceinline__ float entry(int k) const {
    return tok * (row_scale[k] * code_scale) * limb_sum(v[k], v[stride + k], v[2 * stride + k], v[3 * stride + k]);
  }
  __device__ __forceinline__ float& home(int k) const { return *reinterpret_cast<float*>(v + k); }
};

// The norm kernels, one CTA per token.  An entry is fetched once, by a thread that keeps it in shared memory (past kVecKept
// entries: at its home); the squares are added as kVecThreads threads take them whatever the block, which fixes the order of
// that sum.  Bound by their own latency, a part of which is the fetch of their instructions: the loops are hardly unrolled.
// (Split kernel alone, r = 64 / 896 / 1024 / 2048: 2.1 / 3.3 / 3.0 / 4.2 us, the last three from 10, 9 and 4 runs; with a thread's
// entries in eight registers and every loop over them unrolled 2.4 / 5.4 / 4.8 / 3.6, with blocks of 256 2.1 / 5.8 / 4.4 / 9.4.)
constexpr int kVecThreads = 256, kVecMaxThreads = 1024, kVecKept = 4096;
inline int vec_threads(int r) { return r <= 256 ? 256 : r <= 512 ? 512 : kVecMaxThreads; }
template <typename Vec>
struct Kept {
  const Vec& vec;
  float* sm;
  int room;  // entries of sm
  __device__ __forceinline__ float get(int k) const { return k < room ? sm[k] : vec.home(k); }
  __device__ __forceinline__ void put(int k, float e) const {
    if (k < room) sm[k] = e;
    else vec.home(k) = e;
  }
};
// Fetches the entries (thread k mod blockDim.x's are there for itself) and returns 1 / rms, or 1.  ONE: a block of kVecThreads
// for at most as many entries.
template <bool ONE, typename Vec>
__device__ __forceinline__ float take_vec(const Kept<Vec>& v, int r, float eps, int use_rms, float* red) {
  const int tid = threadIdx.x;
  float ss = 0.f;
  if (ONE) {
    const float e = tid < r ? v.vec.entry(tid) : 0.f;
    ss = e * e;
    v.put(tid, e);
  } else {
#pragma unroll 2
    for (int k = tid; k < r; k += blockDim.x) {
      const float e = v.vec.entry(k);
      ss = fmaf(e, e, ss);
      v.put(k, e);
    }
  }
  if (!use_rms) return 1.f;
  if (!ONE && blockDim.x != kVecThreads) {
    __syncthreads();
    ss = 0.f;
    if (tid < kVecThreads)
#pragma unroll 4
      for (int k = tid; k < r; k += kVecThreads) ss = fmaf(v.get(k), v.get(k), ss);
  }
  if (ONE || tid < kVecThreads) {
    ss = warp_sum(ss);
    if ((tid & 31) == 0) red[tid >> 5] = ss;
  }
  __syncthreads();
  float tot = 0.f;
#pragma unroll
  for (int w = 0; w < kVecThreads / 32; ++w) tot += red[w];
  return rsqrtf(tot / (float)r + eps);
}
__device__ __forceinline__ float normed(float e, float inv, const float* gain, int use_rms, int k) {
  return use_rms ? (gain ? gain[k] : 1.f) * e * inv : e;
}

// LoPA gate, batched: n = RMSNorm(v) (or v itself) as a sum of two bf16 vectors for the tensor cores: row b of
// x2 holds the high part of token b's vector, row cols + b the low part (v - bf16(v)), so that the gate's U n keeps
// close to fp32 accuracy.  `exact`: row 2 cols + b holds what those two leave (24 bits in all).
template <bool ONE>
__global__ void __launch_bounds__(ONE ? kVecThreads : kVecMaxThreads) rmsnorm_split_kernel(SumVec vec, int r, const float* gain, float eps, int use_rms,
                                                                       int cols, int exact, __nv_bfloat16* x2) {
  constexpr int kRoom = ONE ? kVecThreads : kVecKept;
  __shared__ float kept[kRoom], red[kVecThreads / 32];
  pdl_launch_dependents();
  pdl_wait();
  const int b = blockIdx.x;
  vec.token(b);
  const Kept<SumVec> v{vec, kept, kRoom};
  const float inv = take_vec<ONE>(v, r, eps, use_rms, red);
#pragma unroll 1
  for (int k = threadIdx.x; k < r; k += ONE ? kVecThreads : blockDim.x) {
    float n = normed(v.get(k), inv, gain, use_rms, k);
    x2[(size_t)b * r + k] = take_bf16(n);
    x2[(size_t)(cols + b) * r + k] = take_bf16(n);
    if (exact) x2[(size_t)(2 * cols + b) * r + k] = __float2bfloat16(n);
  }
}

// Tokens as int8 limbs for the kind::i8 MMAs: t[k] = scale * (q0 + q1 / 128 + q2 / 128^2 + q3 / 128^3) up to
// scale * 2^-22, with scale = max |t| / 127, |q0| <= 127 and the other limbs <= 64 in magnitude.  Row 4 b + l of
// `limbs` holds limb l of token b.  One CTA per token.
// scale of a token whose threads have seen entries of at most m
__device__ __forceinline__ float limb_scale(float m, float* red) {
#pragma unroll
  for (int d = 16; d >= 1; d >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, d));
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = m;
  __syncthreads();
  float mx = 0.f;
  for (int w = 0; w < blockDim.x / 32; ++w) mx = fmaxf(mx, red[w]);
  return mx > 0.f ? mx / 127.f : 1.f;
}
// the limbs of one entry
__device__ __forceinline__ void limbs_of(float e, float inv, int* q4) {
  float t = fminf(fmaxf(e * inv, -127.f), 127.f);
#pragma unroll
  for (int l = 0; l < 4; ++l) {
    const float q = rintf(t);
    q4[l] = (int)q;
    t = (t - q) * 128.f;
  }
}

// A thread takes N consecutive entries at a time, stores N limbs at a time and keeps its first entries, which are all there are up
// to N * 1024 columns.  Bound by its own latency, which stands between the predecessor and the first gate MMA: one round trip to
// the token instead of two dozen (4096 entries by 256 threads, an entry at a time, twice: calls of 4096 x 14336 with 2 to 64
// tokens 8 to 9 us longer, of 8192 x 24000 20 us).
constexpr int kLimbMaxThreads = 1024;
template <int N>
struct LimbGroup;
template <>
struct LimbGroup<8> {
  using In = uint4;
  using Out = uint2;
};
template <>
struct LimbGroup<2> {
  using In = uint32_t;
  using Out = uint16_t;
};
template <int N>
__global__ void __launch_bounds__(kLimbMaxThreads) token_limbs_kernel(const __nv_bfloat16* x, int K, int x_stride, int8_t* limbs,
                                                                      float* scale, int4* zero, int zero_n) {
  using In = typename LimbGroup<N>::In;
  using Out = typename LimbGroup<N>::Out;
  union Entries {
    In in;
    __nv_bfloat16 e[N];
    __device__ Entries() : in() {}
  };
  union Limbs {
    Out out;
    int8_t q[N];
    __device__ Limbs() : out() {}
  };
  __shared__ float red[kLimbMaxThreads / 32];
  pdl_launch_dependents();
  pdl_wait();
  const int b = blockIdx.x, tid = threadIdx.x;
  const In* xb = reinterpret_cast<const In*>(x + (size_t)b * x_stride);
  const int n = K / N;
  Entries first;
  if (tid < n) first.in = xb[tid];
  for (int k = tid; k < zero_n; k += blockDim.x) zero[(size_t)b * zero_n + k] = make_int4(0, 0, 0, 0);
  float m = 0.f;
  auto largest = [&](const Entries& w) {
#pragma unroll
    for (int q = 0; q < N; ++q) m = fmaxf(m, fabsf(__bfloat162float(w.e[q])));
  };
  Entries w = first;
#pragma unroll 1
  for (int k = tid; k < n; w.in = xb[k]) {
    largest(w);
    if ((k += blockDim.x) >= n) break;
  }
  const float s = limb_scale(m, red);
  if (tid == 0) scale[b] = s;
  const float inv = 1.f / s;
  int8_t* out = limbs + (size_t)4 * b * K;
  w = first;
#pragma unroll 1
  for (int k = tid; k < n; w.in = xb[k]) {
    Limbs o[4];
#pragma unroll
    for (int q = 0; q < N; ++q) {
      int l4[4];
      limbs_of(__bfloat162float(w.e[q]), inv, l4);
#pragma unroll
      for (int l = 0; l < 4; ++l) o[l].q[q] = (int8_t)l4[l];
    }
#pragma unroll
    for (int l = 0; l < 4; ++l) *reinterpret_cast<Out*>(out + (size_t)l * K + N * k) = o[l].out;
    if ((k += blockDim.x) >= n) break;
  }
}

// LoPA gate with rows of codes: n = RMSNorm(v) (or v itself) as limbs.
template <bool ONE, typename Vec>
__global__ void __launch_bounds__(ONE ? kVecThreads : kVecMaxThreads) rmsnorm_limbs_kernel(Vec vec, int r, const float* gain, float eps, int use_rms,
                                                                       int8_t* limbs, float* scale) {
  constexpr int kRoom = ONE ? kVecThreads : kVecKept;
  __shared__ float kept[kRoom], red[kVecThreads / 32], red2[kVecMaxThreads / 32];
  pdl_launch_dependents();
  pdl_wait();
  const int b = blockIdx.x;
  vec.token(b);
  const Kept<Vec> v{vec, kept, kRoom};
  const float inv_rms = take_vec<ONE>(v, r, eps, use_rms, red);
  float m = 0.f;
#pragma unroll 1
  for (int k = threadIdx.x; k < r; k += blockDim.x) m = fmaxf(m, fabsf(normed(v.get(k), inv_rms, gain, use_rms, k)));
  const float s = limb_scale(m, red2);
  if (threadIdx.x == 0) scale[b] = s;
  const float inv = 1.f / s;
#pragma unroll 1
  for (int k = threadIdx.x; k < r; k += blockDim.x) {
    int q4[4];
    limbs_of(normed(v.get(k), inv_rms, gain, use_rms, k), inv, q4);
#pragma unroll
    for (int l = 0; l < 4; ++l) limbs[((size_t)4 * b + l) * r + k] = (int8_t)q4[l];
  }
}

}  // namespace


// Tiling of the gate GEMM over R rows (the up kernel needs it to read the gate's bit masks).
void umma_gate_tiling(int R, int K, int qbits, int B, int sm_count, int* tile_rows, int* n_tiles) {
  const int grid = R < 8 * sm_count ? (R + 7) / 8 : sm_count;
  *tile_rows = tile_rows_for(R, grid, equal_tiles_max(K, qbits, B));
  *n_tiles = (R + *tile_rows - 1) / *tile_rows;
}

bool umma_own_list_supported(int R, int K, int qbits, int B, int sm_count) {
  int tr, nt;
  umma_gate_tiling(R, K, qbits, B, sm_count, &tr, &nt);
  return nt <= kThreadsRows && R <= (long long)kMaxOwnTiles * kTileRows * sm_count;
}

bool umma_may_walk(int B) { return B >= kWalkMinTokens; }

bool umma_rows_supported(int K, int cols) { return K % kAtomK == 0 && K >= kAtomK && cols >= 1 && cols <= kUmmaMaxCols; }
// int8 rows multiplied as int8 (tokens as four int8 limbs each): K blocks of 128 codes, up to 64 tokens.
bool umma_rows_native_i8_supported(int K, int tokens) { return K % 128 == 0 && K >= 128 && tokens >= 1 && tokens <= 64; }

namespace {

typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

EncodeTiledFn encode_fn() {
  static EncodeTiledFn fn = nullptr;
  if (!fn) {
    cudaDriverEntryPointQueryResult q;
    void* ptr = nullptr;
    if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &ptr, cudaEnableDefault, &q) == cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = reinterpret_cast<EncodeTiledFn>(ptr);
  }
  return fn;
}

// bf16 matrix [rows, K] with row pitch `pitch_elems`, read in boxes of 64 elements x box_rows rows, 128-byte swizzle.
bool make_map(CUtensorMap* m, const void* base, int K, int rows, size_t pitch_elems, int box_rows) {
  EncodeTiledFn fn = encode_fn();
  if (!fn) return false;
  const cuuint64_t dims[2] = {(cuuint64_t)K, (cuuint64_t)rows};
  const cuuint64_t strides[1] = {(cuuint64_t)pitch_elems * 2};
  const cuuint32_t box[2] = {(cuuint32_t)kAtomK, (cuuint32_t)box_rows};
  const cuuint32_t estr[2] = {1, 1};
  return fn(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(base), dims, strides, box, estr,
            CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// Rows of weight codes [rows, K] (qbits 8 or 4 per code, `pitch_bytes` apart), read in boxes of 64 codes x box_rows
// rows that land densely, without swizzle.
bool make_map_codes(CUtensorMap* m, const void* base, int K, int rows, size_t pitch_bytes, int box_rows, int qbits,
                    int box_codes = kAtomK) {
  EncodeTiledFn fn = encode_fn();
  if (!fn) return false;
  const cuuint64_t dims[2] = {(cuuint64_t)K * qbits / 8, (cuuint64_t)rows};
  const cuuint64_t strides[1] = {(cuuint64_t)pitch_bytes};
  const cuuint32_t box[2] = {(cuuint32_t)(box_codes * qbits / 8), (cuuint32_t)box_rows};
  const cuuint32_t estr[2] = {1, 1};
  return fn(m, CU_TENSOR_MAP_DATA_TYPE_UINT8, 2, const_cast<void*>(base), dims, strides, box, estr,
            CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// int8 matrix [rows, K] (row pitch in bytes), read in boxes of 128 codes x box_rows rows, 128-byte swizzle: the operand
// layout of the kind::i8 MMAs.
bool make_map_i8(CUtensorMap* m, const void* base, int K, int rows, size_t pitch_bytes, int box_rows) {
  EncodeTiledFn fn = encode_fn();
  if (!fn) return false;
  const cuuint64_t dims[2] = {(cuuint64_t)K, (cuuint64_t)rows};
  const cuuint64_t strides[1] = {(cuuint64_t)pitch_bytes};
  const cuuint32_t box[2] = {128u, (cuuint32_t)box_rows};
  const cuuint32_t estr[2] = {1, 1};
  return fn(m, CU_TENSOR_MAP_DATA_TYPE_UINT8, 2, const_cast<void*>(base), dims, strides, box, estr,
            CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

bool make_weight_map(CUtensorMap* m, const void* base, int K, int rows, int box_rows, int qbits) {
  return qbits == 1 ? make_map_i8(m, base, K, rows, (size_t)K, box_rows)
         : qbits == 2 ? make_map_codes(m, base, K, rows, (size_t)K / 2, box_rows, 4, 128)  // int4 rows, K blocks of 128 codes
         : qbits    ? make_map_codes(m, base, K, rows, (size_t)K * qbits / 8, box_rows, qbits)
                    : make_map(m, base, K, rows, (size_t)K, box_rows);
}

template <int MODE, typename Map>
cudaError_t launch_rows_mode(const UmmaRowsParams& p, dim3 grid, size_t smem, cudaStream_t s, const CUtensorMap& map_w,
                             const CUtensorMap& map_x, const Map& map_t) {
  static unsigned long long configured[4] = {0, 0, 0, 0};
  cudaError_t e;
  if constexpr (MODE != kUpMayWalk) {
    if (p.exact) {
      static unsigned long long configured_ex[3] = {0, 0, 0};
      auto k = p.qbits == 8 ? umma_rows_kernel<MODE, 8, true> : p.qbits == 4 ? umma_rows_kernel<MODE, 4, true> : umma_rows_kernel<MODE, 0, true>;
      if ((e = allow_dynamic_smem(k, 227 * 1024, configured_ex[p.qbits == 8 ? 1 : p.qbits == 4 ? 2 : 0])) != cudaSuccess) return e;
      return launch_pdl(k, grid, dim3(kThreadsRows + 128 + (p.qbits ? 32 * kExpandWarps : 0)), smem, s, p, map_w, map_x, map_t);
    }
  }
  if constexpr (MODE != kUp) {
    if (p.pair) {
      static unsigned long long configured_pair[2] = {0, 0};
      auto k = p.qbits ? umma_rows_kernel<MODE, 1, false, true> : umma_rows_kernel<MODE, 0, false, true>;
      if ((e = allow_dynamic_smem(k, 227 * 1024, configured_pair[p.qbits])) != cudaSuccess) return e;
      return launch_clusters(2, k, grid, dim3(kThreadsRows), smem, s, p, map_w, map_x, map_t);
    }
  }
  if (p.qbits == 1) {
    auto k = umma_rows_kernel<MODE, 1>;
    if ((e = allow_dynamic_smem(k, 227 * 1024, configured[3])) != cudaSuccess) return e;
    return launch_pdl(k, grid, dim3(kThreadsRows), smem, s, p, map_w, map_x, map_t);
  }
  if (p.qbits == 2) {
    static unsigned long long configured2[2] = {0, 0};
    const bool tall = p.K > kShortRow && tile_rows_for(p.R, grid.x, p.equal_max) > kTallTile;
    auto k = tall ? umma_rows_kernel<MODE, 3> : umma_rows_kernel<MODE, 2>;
    if ((e = allow_dynamic_smem(k, 227 * 1024, configured2[tall])) != cudaSuccess) return e;
    return launch_pdl(k, grid, dim3(kThreadsRows + 32 * kExpandWarps), smem, s, p, map_w, map_x, map_t);
  }
  if (p.qbits == 8) {
    auto k = umma_rows_kernel<MODE, 8>;
    if ((e = allow_dynamic_smem(k, 227 * 1024, configured[0])) != cudaSuccess) return e;
    return launch_pdl(k, grid, dim3(kThreadsRows + 32 * kExpandWarps), smem, s, p, map_w, map_x, map_t);
  }
  if (p.qbits == 4) {
    auto k = umma_rows_kernel<MODE, 4>;
    if ((e = allow_dynamic_smem(k, 227 * 1024, configured[1])) != cudaSuccess) return e;
    return launch_pdl(k, grid, dim3(kThreadsRows + 32 * kExpandWarps), smem, s, p, map_w, map_x, map_t);
  }
  auto k = umma_rows_kernel<MODE, 0>;
  if ((e = allow_dynamic_smem(k, 227 * 1024, configured[2])) != cudaSuccess) return e;
  return launch_pdl(k, grid, dim3(kThreadsRows), smem, s, p, map_w, map_x, map_t);
}

}  // namespace

// The LoPA stage v = V x has few rows (the rank) of many columns.  A tile of eight rows for each SM reads all token columns for
// them: with tiles of up to 64 rows and K cut into runs all CTAs together read an eighth of that, and ranks below 8 rows per SM
// fill the SMs too.  The next kernel adds the fp32 sums of the runs in their order; integer sums (limbs) are added in memory, so
// that what cancels across runs leaves nothing behind and v has the bits of one run (as int4 of every run, added by the norm,
// calls of r >= 1280 were 2 us longer: one SM read 130 KB).  Whole calls, power-law firing, not cut / cut: 4096 x 14336, r = 512,
// 4 / 64 tokens, bf16 46.2 / 94.3 -> 44.5 / 86.8 us, int4 44.2 / 108 -> 42.1 / 97.7; 8192 x 28672, r = 1024, 8 tokens, int8
// 101 -> 95.7.
// Rows of up to kShortRow columns are cut from 16 tokens on: fewer hand little over, and the cut costs the norm more round trips
// (1024 x 3000, r = 128, 2 / 8 / 16 / 64 tokens, not cut / cut: bf16 25.5 / 28.4 / 29.9 / 42.8 us against 26.4 / 28.5 / 30.0 / 41.3;
// int4 29.6 / 32.9 / 36.4 / 56.6 against 29.8 / 32.6 / 35.4 / 55.5).  The runs differ by at most one block of K.
void umma_k_splits(int R, int K, bool codes, int B, int sm_count, int max_splits, int* tiles, int* splits) {
  const int kb = K / (codes ? 128 : kAtomK);
  auto least = [](int a, int b) { return a < b ? a : b; };
  int t = (R + 63) / 64, n = least(least(max_splits, 16), least(sm_count / t, kb / 4));
  *tiles = *splits = 1;
  if (n < 2 || (K <= kShortRow && B < 16)) return;
  if (4 * t * n < 3 * sm_count) t = least((R + 7) / 8, sm_count / n);
  const int rows = ((R + t - 1) / t + 7) & ~7;
  *tiles = (R + rows - 1) / rows;
  *splits = n;
}

// Pairs of CTAs (cta_group::2) where a CTA by itself has fewer than six ring slots: each holds half of the token rows, which every
// CTA reads through L2 otherwise, and the ring gets eight slots instead of four.  4096 x 14336, alone / in pairs: bf16, 200 and
// 256 tokens 130 / 112 and 137 / 122 us; int8, 48 and 64 tokens 75.3 / 69.3 and 80.5 / 75.9; 8192 x 24000: 394 / 348, 235 / 210.
// With six slots nothing is gained (4096 x 14336, 160 tokens 99.9 / 100.7; 2048 x 6000, 200 tokens 59.7 / 61.6), and the clusters
// cost a kernel 0.5 to 1 us (1024 x 3000, 72 tokens 29.7 / 33.3).  Codes that are expanded stay alone (int4, 4096 x 14336, 64
// tokens 97.5 / 112: two CTAs' expansions to wait for).
// The up projection goes by R, as the list's length is known on the device alone: time alone over time in pairs, Zipf firing, bf16 176 to
// 256 and int8 40 to 64 tokens, 1024 to 8192 columns, at 10 / 3 / 1.5 / 0.5 / 0.1 % firing 0.98-1.09 / 0.98-1.09 / 0.96-1.13 /
// 0.96-1.10 / 0.92-1.01.
bool umma_rows_pairs(int R, int K, int qbits, int B, int cols, bool exact, int sm_count) {
  if (exact || qbits > 1 || sm_count % 2) return false;
  int tile_rows, n_tiles;
  umma_gate_tiling(R, K, qbits, B, sm_count, &tile_rows, &n_tiles);
  return kRingBytes / ((tile_rows + (cols + 15) / 16 * 16) * 128) < 6;
}

int umma_gate_rows_per_word(int R, int K, int qbits, int B, int cols, bool exact, int sm_count) {
  int tile_rows, n_tiles;
  umma_gate_tiling(R, K, qbits, B, sm_count, &tile_rows, &n_tiles);
  return tile_rows <= 64 && !umma_rows_pairs(R, K, qbits, B, cols, exact, sm_count) ? 16 : 32;
}

cudaError_t launch_umma_rows(bool up, UmmaRowsParams p, int cols, int sm_count, cudaStream_t s) {
  p.npad = (cols + 15) / 16 * 16;
  if (p.exact ? (p.B > (p.qbits ? kExactHalfTerms + 16 : kExactTokens) || p.npad > kUmmaExactCols || p.qbits == 1 || p.qbits == 2 || (up && p.h_terms != 3))
              : p.h_terms > 1 && !(up && p.h_terms == 2 && (p.qbits == 8 || p.qbits == 4))) return cudaErrorInvalidValue;
  if (p.x_cols && (p.x_cols % 8 || cols != (p.exact ? 3 : 2) * p.x_cols)) return cudaErrorInvalidValue;
  p.wait_cycles = fused_test_knobs().wait_cycles;
  p.drop_stage = fused_test_knobs().drop_stage;
  const int splits = p.k_splits > 1 ? p.k_splits : 1;
  if (splits > 1 && (up || p.exact || p.b_g || p.g_idx || p.flag || p.words_out || p.act != kUmmaActIdentity)) return cudaErrorInvalidValue;
  const int kb = p.K / (p.qbits == 1 || p.qbits == 2 ? 128 : kAtomK);
  p.equal_max = equal_tiles_max(p.K, p.qbits, p.B);
  p.run_blocks = kb / splits;
  p.longer_runs = kb % splits;
  const bool may_walk = up && p.walk_all && umma_may_walk(p.B) && !p.exact;
  int grid = splits > 1 ? p.k_tiles : p.R < 8 * sm_count ? (p.R + 7) / 8 : sm_count;
  p.pair = splits == 1 && (!up || may_walk) && umma_rows_pairs(p.R, p.K, p.qbits, p.B, cols, p.exact, sm_count);
  grid += p.pair ? grid % 2 : 0;  // (one CTA more of eight rows each: the same tiles)
  if (p.pair && p.qbits) p.npad = (p.npad + 31) / 32 * 32;  // what the pairs' int8 MMAs take
  // all the dynamic shared memory a CTA can have; the kernel cuts its ring out of it once it knows its tiles
  const size_t smem = kRowsSmem;
  p.ring_bytes = kRingBytes;
  alignas(64) CUtensorMap map_w, map_x;
  if (p.qbits != 0 && p.qbits != 8 && p.qbits != 4 && p.qbits != 1 && p.qbits != 2) return cudaErrorInvalidValue;
  const bool i8 = p.qbits == 1 || p.qbits == 2;  // kind::i8 MMAs: X holds the tokens' int8 limbs
  if (p.npad > kUmmaMaxCols) return cudaErrorInvalidValue;
  if (i8 && (p.K % 128 || !p.tok_scale)) return cudaErrorInvalidValue;
  // weights: all R rows; boxes of one tile's rows for the gate, single-row boxes for the gather
  if (!make_weight_map(&map_w, p.W, p.K, p.R, up ? 1 : tile_rows_for(p.R, grid, p.equal_max), p.qbits)) return cudaErrorNotSupported;
  // tokens: only the rows that exist; the box covers npad rows (half of them in each CTA of a pair) and the rest reads as zero
  const int x_box = p.pair ? p.npad / 2 : p.npad;
  if (i8 ? !make_map_i8(&map_x, p.X, p.K, p.ncols_valid, (size_t)p.x_stride, x_box)
                   : !make_map(&map_x, p.X, p.K, p.ncols_valid, (size_t)p.x_stride, x_box))
    return cudaErrorNotSupported;
  if (!up) return launch_rows_mode<kGate>(p, dim3(grid, splits), smem, s, map_w, map_x, WalkMap<false>{});
  if (may_walk) {
    // wide batches: the union may cover most rows; the kernel then walks every row with tiled boxes of the tile
    // height of R rows (decided on the device from the union's size, so it depends on this call's inputs only)
    WalkMap<true> map_t;
    if (!make_weight_map(&map_t.m, p.W, p.K, p.R, tile_rows_for(p.R, grid, p.equal_max), p.qbits)) return cudaErrorNotSupported;
    return launch_rows_mode<kUpMayWalk>(p, dim3(grid), smem, s, map_w, map_x, map_t);
  }
  return launch_rows_mode<kUp>(p, dim3(grid), smem, s, map_w, map_x, WalkMap<false>{});
}

// Token columns up to which two CTAs of the down kernel share an SM (each with two accumulators in half of the TMEM, and
// at least four ring stages); wider batches give one CTA the whole SM, and so do exact sums, whose accumulators fill
// the TMEM.
constexpr int kDownPairCols = 64;
constexpr int kMaxDownCluster = 8;  // CTAs of a cluster
static bool down_pairs(int cols, bool exact) { return cols <= kDownPairCols && !exact; }

// Clusters of `size` CTAs of the down kernel that the device runs at once, two CTAs per SM or one.  Asked for a kernel that does
// nothing in as many threads and as much shared memory: for one that allocates TMEM the runtime answers as if an SM took a single CTA.
static __global__ void __launch_bounds__(down_bound(8, false), 2) down_place_kernel() {}
static int down_clusters(int dev, int size, bool pairs) {
  static unsigned long long configured = 0;
  static std::atomic<int> known[2][kMaxDownCluster + 1][kKnownDevices];
  return clusters_at_once(dev, down_place_kernel, size, down_bound(8, false), (pairs ? 111 : 225) * 1024, configured, known[pairs][size]);
}

// Splits of the list, and whether they are a cluster that adds its sums up itself.  That saves the partials' way through memory and
// a kernel (4096 x 14336, bf16, short runs, partials / clusters: 200 tokens 108.3 / 101.2 us, 72 tokens 83.3 / 79.4, 16 tokens 62.9 / 61.6; 512 x
// 1500, int8, 2 tokens 21.5 / 18.9), and costs splits where more CTAs would run than clusters fit the GPCs.  Clusters:
// - where they cost up to a ninth of the splits (codes, whose blocks take longer: none): int8, 4096 x 14336, 8 tokens, nine splits /
//   clusters of eight 44.6 / 45.1; bf16, 6144 x 20000, 160 tokens, three / two 229 / 242;
// - or any number of them where a CTA has few blocks.  A dozen where the list has codes, or the fired rows of up to eight tokens (2048 x
//   6144, 16 / 8: int4, 2 / 24 / 64 tokens 26.7 / 36.9 / 50.7 against 24.4 / 37.6 / 49.0; bf16, 2 tokens 25.7 / 25.2; codes of 16 to 32
//   tokens between 65 and 96 blocks: from 6 % slower to 4 % faster), else eight (bf16, 16 / 8, 63 blocks: 1024 x 3993, 16 / 32 / 64
//   tokens 22.5 / 24.8 / 29.9 against 23.2 / 23.8 / 28.7; 72 blocks: 1536 x 4608, 16 / 24 / 64 tokens 26.9 / 26.8 / 33.3 against 28.4 /
//   28.7 / 33.9).
// Clusters of an odd size need a sixteenth of room to spare: they split the two SMs of a TPC, and the SMs that the kernel before leaves
// one after the other do not always come to as many clusters as an empty device takes (tiles / most that fit at once, partials /
// clusters: 42 / 45 of three, 5376 x 16128, bf16, 100 tokens 115 / 111 us, but 45 / 45, 5760 x 17280, int8, 100 tokens 179 / 227; 52 /
// 56 of five, 6656 x 19968, bf16, 24 tokens 139 / 137, but 56 / 56, 7168 x 21504, int8 122 / 145).  Clusters of up to 16 where they fit
// are slower (512 x 1500, bf16, 24 tokens, 8 / 16: 19.4 / 20.4).
// Exact sums: three blocks a CTA, or six for up to 24 tokens (three columns each); their CTAs work longer on each block, and the sum has
// less to hide (partials / clusters of eight: 384 x 1152, bf16, 6 / 64 tokens 34.4 / 59.2 against 31.7 / 59.1; 640 x 1920, 6 / 24 / 64
// tokens 35.1 / 40.3 / 67.3 against 33.9 / 39.9 / 69.0; 896 x 2688, 64 / 256 tokens 77.6 / 320 against 81.3 / 336; 1152 x 3287, 13 tokens
// 43.4 / 44.4; of three, 43 tiles: 5504 x 16512, 6 / 15 tokens 163 / 206 against 170 / 233).
constexpr int kExactClusterCols = 72;
bool umma_down_splits(int D, int R, int qbits, int cols, bool exact, int sm_count, int max_splits, int* splits, const int* at_once) {
  const int tiles = D >= kTileRows ? D / kTileRows : 1;
  const bool pairs = down_pairs(cols, exact);
  const int dev = at_once ? -1 : current_device();
  int cluster = kMaxDownCluster;
  auto fits = [&](int size) {
    const int most = at_once ? at_once[size] : down_clusters(dev, size, pairs);
    return most >= tiles && (size % 2 == 0 || 15 * most >= 16 * tiles);
  };
  while (cluster > 1 && !fits(cluster)) --cluster;
  auto splits_of = [&](int ctas) {
    const int n = ctas / tiles;
    return n < 1 ? 1 : n > max_splits ? max_splits : n;
  };
  const int one = splits_of(sm_count), two = splits_of(2 * sm_count);
  int n = pairs ? two : one;
  // Exact sums: two waves of CTAs, each with a set-up of its own (about 6 us), only where they shorten the contraction by a
  // tenth: wide rows, whose tiles leave SMs idle in one wave.  16 tokens, one wave / two: 2688 x 8000 67 / 74 us, 6528 x
  // 20000 (102 and 255 CTAs) 312 / 301.
  if (exact && 10 * (two - 2 * one) >= one * two) n = two;
  const int blocks = (R + kAtomK - 1) / kAtomK;
  if (exact && n == 1) cluster = 1;
  const bool clustered = exact ? n == 1 : qbits ? cluster >= n : 9 * cluster >= 8 * n;
  const int few = (exact ? (cols <= kExactClusterCols ? 6 : 3) : qbits || cols <= 8 ? 12 : 8) * cluster;
  if (clustered || (cluster > 1 && blocks <= few)) {
    *splits = cluster;
    return true;
  }
  *splits = n;
  return false;
}

bool umma_down_supported(int D, int cols) { return D % kTileRows == 0 && cols >= 1 && cols <= kUmmaMaxCols; }

namespace {
template <int QB, bool EX = false, bool TWO = false, bool CL = true>
cudaError_t launch_down_q(const UmmaDownParams& p, int grid, size_t smem, cudaStream_t s, const CUtensorMap& map_wg,
                          const CUtensorMap& map_wt, const CUtensorMap& map_hm) {
  static unsigned long long configured = 0;
  const cudaError_t e = allow_dynamic_smem(umma_down_kernel<QB, EX, TWO, CL>, 227 * 1024, configured);
  if (e != cudaSuccess) return e;
  return launch_clusters(p.y ? p.splits : 1, umma_down_kernel<QB, EX, TWO, CL>, dim3(grid), dim3((EX ? 512 : kThreads) + (QB ? 32 * kExpandWarps : 0)), smem, s, p, map_wg,
                    map_wt, map_hm);
}
}  // namespace

cudaError_t launch_umma_down(UmmaDownParams p, cudaStream_t s) {
  if (p.qbits != 0 && p.qbits != 8 && p.qbits != 4) return cudaErrorInvalidValue;
  if (p.terms < 1) p.terms = 1;
  if (p.exact ? p.terms != 3 || p.cols > kExactTokens || p.npad > kUmmaExactCols : p.terms > 2 || (p.terms == 2 && !p.qbits)) return cudaErrorInvalidValue;
  const int own = p.terms * p.cols;  // token columns that carry something
  p.npad = (own + 15) / 16 * 16;
  if (p.cols % 8 || p.cols < p.B || p.npad > kUmmaMaxCols) return cudaErrorInvalidValue;
  p.wait_cycles = fused_test_knobs().wait_cycles;
  const int room = (down_pairs(own, p.exact) ? 111 : 225) * 1024 - 1024 - 1024;
  const int copies = p.npad * 128 + p.qbits * kTileRows * kAtomK / 8;  // of a stage: h, and the codes of quantised rows
  // Codes: no more slots than a CTA has blocks of 64 rows, so that narrow models, whose many splits get a block or two, keep
  // one ring (the second one's barriers and hand-overs: 0.3 us of 6.3 at 256 columns).
  const int blocks = ((p.R + kAtomK - 1) / kAtomK + p.splits - 1) / p.splits;
  const int most = !p.qbits || p.exact || blocks > 12 ? 12 : (blocks + 1) & ~1;
  auto slots = [&](int expand) {  // ring slots beside `expand` expanded blocks, or with a block each (0)
    const int n = (room - expand * kAAtomBytes) / (copies + (expand ? 0 : kAAtomBytes));
    return (n > most ? most : n) & (p.exact ? ~3 : ~1);
  };
  // Expanded blocks: two leave more slots for the copies, which is worth more (int8, 4096 x 14336, 16 tokens, 2 / 4: 56.9 / 58.1
  // us), but four where a CTA has the SM to itself and four slots are left (int8, 4480 x 13000, 64 tokens, 6 slots: 114 / 110;
  // 128 tokens, where they leave two slots: 147 / 167).
  p.expand = !down_pairs(own, p.exact) && slots(kDownExpand) >= 4 ? kDownExpand : 2;
  // One ring where it has six slots or no fewer than two rings would, and for 4-bit codes that are walked rather than gathered
  // (from 32 tokens on) where it has four: nothing is left to gain, and a block for each slot keeps the expansion further ahead
  // (one ring / two: int8, 4480 x 13000, 48 and 96 tokens 105.5 / 107.0 and 121.1 / 121.9 us; int4, 40 and 128 tokens 109.0 /
  // 110.0 and 130.9 / 131.8; int4, 8192 x 18000, 32 tokens 152.7 / 156.4, but 24 tokens 131.6 / 124.7).
  const bool two = p.qbits && !p.exact && slots(0) < 6 && slots(p.expand) > slots(0) &&
                   !(p.qbits == 4 && p.B >= kWalkMinTokens && slots(0) >= 4);
  const int expanded = two ? p.expand * kAAtomBytes : 0;
  const int stage_bytes = copies + (two ? 0 : kAAtomBytes);
  const int stages = slots(two ? p.expand : 0);
  if (stages < 2) return cudaErrorInvalidValue;
  p.stages = stages;
  p.ring_bytes = expanded + stages * stage_bytes;
  if (p.ring_bytes < p.cols * kTileRows * 4) p.ring_bytes = p.cols * kTileRows * 4;
  size_t smem = 1024 + p.ring_bytes + (3 * stages + 4 + 2 * kMaxIssuers + 2 * kDownExpand) * 8 + 64;
  // Never so little that an SM takes more CTAs than its TMEM has room for: they would wait for it (int8, 640 x 1408, 87 tokens:
  // 36.5 -> 39.8 us).
  const size_t least = (down_pairs(own, p.exact) ? 80 : 120) * 1024;
  if (smem < least) smem = least;
  const int grid = (p.D / kTileRows) * p.splits;
  alignas(64) CUtensorMap map_wg, map_wt, map_hm;
  // W_down [H, D]: inner dimension d; single-row boxes for the gather, 64-row boxes for the dense walk
  if (!make_weight_map(&map_wg, p.W_down, p.D, p.R, 1, p.qbits)) return cudaErrorNotSupported;
  if (!make_weight_map(&map_wt, p.W_down, p.D, p.R, kAtomK, p.qbits)) return cudaErrorNotSupported;
  // HmT [terms * h_cols][hm_stride]: inner dimension u; one box of `cols` token rows per term
  if (!make_map(&map_hm, p.hmT, p.hm_stride, p.terms * p.h_cols, (size_t)p.hm_stride, p.cols)) return cudaErrorNotSupported;
  const int g = grid;
  if (p.exact)
    return p.qbits == 0 ? launch_down_q<0, true>(p, g, smem, s, map_wg, map_wt, map_hm)
           : p.qbits == 8
               ? p.y ? launch_down_q<8, true>(p, g, smem, s, map_wg, map_wt, map_hm) : launch_down_q<8, true, false, false>(p, g, smem, s, map_wg, map_wt, map_hm)
           : p.y ? launch_down_q<4, true>(p, g, smem, s, map_wg, map_wt, map_hm)
                 : launch_down_q<4, true, false, false>(p, g, smem, s, map_wg, map_wt, map_hm);
  if (two)
    return p.qbits == 8 ? launch_down_q<8, false, true>(p, g, smem, s, map_wg, map_wt, map_hm)
                        : launch_down_q<4, false, true>(p, g, smem, s, map_wg, map_wt, map_hm);
  return p.qbits == 8   ? launch_down_q<8>(p, g, smem, s, map_wg, map_wt, map_hm)
         : p.qbits == 4 ? launch_down_q<4>(p, g, smem, s, map_wg, map_wt, map_hm)
                        : launch_down_q<0>(p, g, smem, s, map_wg, map_wt, map_hm);
}

// Pairs of entries up to this many columns: groups of eight leave a token of 256 columns to one warp (whole calls, 256 x 700, 4 /
// 16 tokens, eights / pairs: int4 23.3 / 26.1 us -> 22.3 / 25.4; int8, 768 x 2300, 24 tokens 30.1 -> 29.6).  At 1024 columns pairs
// are 512 threads, beside which an SM has no registers left for a CTA of the 4-bit gate (512 threads of 106), so that it starts
// late where the grid needs that SM (int4, 1024 x 3000, 32 / 40 tokens, pairs / eights: 35.5 / 38.1 -> 34.4 / 37.1).  Longer tokens
// want their threads nevertheless (256 at most instead of 512 at 4096 columns, 1024 at 8192: 1 to 2 % slower).
constexpr int kShortToken = 768;
cudaError_t launch_token_limbs(const void* x, int B, int K, int x_stride, void* limbs, float* scale, void* zero, int zero_bytes,
                               cudaStream_t s) {
  const bool pairs = K <= kShortToken;
  const int groups = (K / (pairs ? 2 : 8) + 31) / 32 * 32;
  return launch_pdl(pairs ? token_limbs_kernel<2> : token_limbs_kernel<8>, dim3(B), dim3(groups < kLimbMaxThreads ? groups : kLimbMaxThreads),
                    0, s, static_cast<const __nv_bfloat16*>(x), K, x_stride, static_cast<int8_t*>(limbs), scale, static_cast<int4*>(zero),
                    zero_bytes / 16);
}

cudaError_t launch_rmsnorm_limbs(float* v, int B, int r, int v_stride, const UmmaLimbSums* sums, const float* gain, float eps,
                                 bool use_rms, void* limbs, float* scale, cudaStream_t s) {
  const dim3 block(vec_threads(r));
  int8_t* out = static_cast<int8_t*>(limbs);
  const bool one = r <= kVecThreads;
  if (!sums) {
    const SumVec vec{v, v_stride, 1, 0};
    return launch_pdl(one ? rmsnorm_limbs_kernel<true, SumVec> : rmsnorm_limbs_kernel<false, SumVec>, dim3(B), block, 0, s, vec, r, gain, eps,
                      use_rms ? 1 : 0, out, scale);
  }
  const LimbSumsVec vec{reinterpret_cast<int*>(v), v_stride, sums->row_scale, sums->tok_scale, sums->code_scale, 0.f};
  return launch_pdl(one ? rmsnorm_limbs_kernel<true, LimbSumsVec> : rmsnorm_limbs_kernel<false, LimbSumsVec>, dim3(B), block, 0, s, vec, r, gain,
                    eps, use_rms ? 1 : 0, out, scale);
}

cudaError_t launch_rmsnorm_split(float* v, int B, int r, int v_stride, int runs, size_t step, const float* gain, float eps,
                                 bool use_rms, int cols, bool exact, void* x2, cudaStream_t s) {
  const SumVec vec{v, v_stride, runs, step};
  return launch_pdl(r <= kVecThreads ? rmsnorm_split_kernel<true> : rmsnorm_split_kernel<false>, dim3(B), dim3(vec_threads(r)), 0, s, vec, r,
                    gain, eps, use_rms ? 1 : 0, cols, exact ? 1 : 0, static_cast<__nv_bfloat16*>(x2));
}

}  // namespace sffn
