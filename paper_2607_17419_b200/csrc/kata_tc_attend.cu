// KATA forward of blocks of 256 queries on the Blackwell tensor cores (tcgen05 + TMEM), bf16: the quadratic
// ("flash-style") form, and the output stage of the chunked form.
//
// Pre-pass (one light kernel per call): r[i] = 1 / ||k_i||^2 (bf16) into the workspace.
//
// Main kernel: persistent, one CTA per SM.  A work item = one head x 256 queries (two tiles of 128: the halves A and B);
// the items are ordered heaviest first and dealt to the CTAs in rounds, forwards and backwards in turn.  An item is a
// list of tiles that both halves walk:
//   state tiles (chunked form, chunks after the first): the state S, Z before the chunk, in bf16
//     [O | D] += Psi(Q) [S | Z]   256 rows of the state per tile; the builders write the 256 feature products of their
//                                 query row as the A operand (TMEM); Z is column 64 of B, so numerator and normaliser
//                                 see the same rounded features (a Z of its own, q . Z q from the fp32 products, left
//                                 rows with a small normaliser outside the bf16 tolerance)
//   key tiles of 128 keys, from the start of the chunk (quadratic form: of the sequence) up to the diagonal:
//     scores   S = Q K_j^T            A = the query tile in TMEM, B = the key tile (TMA, 128B swizzle)
//     weights  P = r S^2 (causal mask on the diagonal tiles)  packed fp32x2 multiplies on the TMEM read-back, rounded
//                                     to bf16, times r, stored back over the scores; with exact key scales (XR) times
//                                     r in fp32 and rounded once
//     apply    [O | D] += P [V | 1]   A = P from TMEM, B = the value tile and a constant column of ones (MN-major,
//                                     N = 80): the normaliser is column 64 of the same accumulator
//   epilogue out = O / D  (0 where that is 0)      the gate/normalise step of the readout
// There is no running maximum and no rescaling: the weights are polynomial.  The query norm cancels between
// numerator and denominator and is never applied.  In the quadratic form the d^2-wide feature state is never formed.
// Rows narrower than 64 entries are read by TMA boxes of 64 columns, whose columns beyond the row are zero; with up to 32
// entries (R = 4 runs of 8) the empty half of the features is left out: 12 block pairs instead of 36, two score steps
// instead of four (8 heads x 16 x 6000 tokens of 32 entries 501 -> 312 us, 16 x 60000 828 -> 486).
//
// The issuers' descriptors are sums of a constant and a stage's offset, and what is checked once an item or a tile is checked
// outside the loop over the sub-buffers: an issuer shares its scheduler with four builder warps, and every instruction of its
// waits a few cycles for a slot (per sub-buffer of 64 keys a wait, 8 MMAs and a commit, some 370 cycles of which the pipe has
// use for 288; 64 heads x 4096 tokens 128.9 -> 124.1 us).
//
// What bounds it and why this split.  A key tile is 576 cycles of MMA per half (4 x N=128, 8 x N=80) and a chain
// scores -> builders -> apply of about 1700, most of it hand-offs.  Four chains run side by side: two halves times two
// sub-buffers of 64 score columns each.  Both halves share every key, value and state tile, which halves the tile
// traffic into shared memory: with one query tile per CTA and Q as a shared-memory operand the port (A and B operands,
// TMA writes, r) was asked for about 800 cycles per key tile, more than the MMAs take; here it is about 480.
//
// Nothing is set up per item: TMEM and the barriers are the CTA's, the stage ring runs on across items (every role
// counts tiles cumulatively), and the next item's query tiles are loaded once the features of this one are built and
// copied to TMEM before its epilogue.
//
// Warps (640 threads): 0 TMA producer, 1 and 2 the MMA issuers of the halves, 3 key scales, 4-11 builders of half A,
// 12-19 builders of half B (TMEM lane quadrant = warp % 4; the two warps of a quadrant have a sub-buffer each).  All
// waits are bounded.
#include <cuda.h>
#include <type_traits>

#include "kata_common.cuh"
#include "kata_pairs.cuh"
#include "kata_tmap.cuh"
#include "kata_umma.cuh"

namespace kata {
namespace {

using namespace umma;

constexpr int D = 64;
constexpr int QT = 128;          // queries per half
constexpr int KTILE = 128;       // score columns per tile
constexpr int NSTAGE = 4;        // shared-memory stages: a key and a value tile, or 256 rows of a state
constexpr int NTHREADS = 640;
constexpr int WARP_BLD0 = 4;

constexpr uint32_t COL_S = 0;    // 2 x 128 fp32 score columns, one buffer per half; the operand of the apply MMA overwrites it
constexpr uint32_t COL_O = 256;  // 2 x 80 fp32 accumulators: 64 outputs, column 64 = normaliser
constexpr uint32_t COL_Q = 416;  // 2 x 32: the query tiles (bf16 A operands)
constexpr uint32_t TMEM_COLS = 512;

constexpr uint32_t OFF_Q = 0;                       // 2 x (128 x 64 bf16, 128B swizzle): the query tiles of an item
constexpr uint32_t STAGE_BYTES = 32768;             // K tile 16 KB, V tile 16 KB
constexpr uint32_t OFF_ST = 32768;
constexpr uint32_t OFF_ONES = OFF_ST + NSTAGE * STAGE_BYTES;   // 16 rows of [1, 0 ...]: columns 64.. of the values
constexpr uint32_t OFF_Z = OFF_ONES + 2048;                    // columns 64.. of a state: 256 rows of 128 bytes, 32 of them per stage
constexpr uint32_t OFF_RV = OFF_Z + 32768;                     // NSTAGE x 128 bf16 or fp32: 1 / ||k||^2 of the keys of a tile
constexpr uint32_t OFF_BAR = OFF_RV + NSTAGE * 512;
constexpr uint32_t SMEM_BYTES = OFF_BAR + 512;
constexpr uint32_t SMEM_ALLOC = SMEM_BYTES + 1024;
static_assert(SMEM_ALLOC > 116 * 1024, "one CTA per SM is assumed (the CTA allocates all of TMEM)");

// No barrier can complete two phases ahead of a waiter; a waiter that skips a phase (the builders the last one of an item
// at BAR_SFREE) knows from a barrier that it waited for since that it is complete.
enum {
  BAR_QFULL = 0,     // the query tiles of an item landed in shared memory
  BAR_QEMPTY = 1,    // ... and have been read (512 builders)
  BAR_FULL = 4,      // [NSTAGE] tile (TMA bytes) and its key scales or Z column (warp 3) landed
  BAR_EMPTY = 8,     // [NSTAGE] stage free: both issuers
  BAR_SFULL = 12,    // [half][sub] scores in TMEM
  BAR_PFULL = 16,    // [half][sub] the builders are done with the sub-buffer (128)
  BAR_FFULL = 20,    // [half][sub][piece] features of a state tile in TMEM (128)
  BAR_SFREE = 28,    // [half][sub][piece] ... and consumed
  BAR_QT = 36,       // [2] query tile in TMEM (128)
  BAR_ODONE = 38,    // [2] the MMAs of an item are complete: [O | D] is final
  BAR_OFREE = 40,    // [2] [O | D] has been read (256): the next item may overwrite it
  BAR_DRAIN = 42,
  BAR_COUNT = 43
};

// Pre-pass: r = 1 / ||k||^2 per key row (0 for a zero row); eight lanes of 16 bytes per row, four rows per lane in flight
// (memory-bound; 33.5 MB of keys: 8.7 us with one row per lane, 6.9 with four).
constexpr int RS_ROWS = 4;
__global__ void __launch_bounds__(256) rscale_kernel(const __nv_bfloat16* __restrict__ k, float* __restrict__ r_f32,
                                                     __nv_bfloat16* __restrict__ r_bf16, size_t n_rows, int d) {
  cudaTriggerProgrammaticLaunchCompletion();   // the kernel behind sets itself up meanwhile
  const size_t row0 = (size_t)blockIdx.x * (32 * RS_ROWS) + (threadIdx.x >> 3);
  const int part = threadIdx.x & 7;
  uint4 raw[RS_ROWS];
#pragma unroll
  for (int i = 0; i < RS_ROWS; ++i) {
    const size_t row = row0 + i * 32;
    raw[i] = make_uint4(0u, 0u, 0u, 0u);
    if (row < n_rows && part * 8 < d) raw[i] = *reinterpret_cast<const uint4*>(k + row * d + part * 8);
  }
#pragma unroll
  for (int i = 0; i < RS_ROWS; ++i) {
    const uint32_t kw[4] = {raw[i].x, raw[i].y, raw[i].z, raw[i].w};
    float ss = 0.f;
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      const float lo = __uint_as_float(kw[e] << 16), hi = __uint_as_float(kw[e] & 0xFFFF0000u);
      ss = fmaf(lo, lo, ss);
      ss = fmaf(hi, hi, ss);
    }
    ss += __shfl_xor_sync(0xffffffffu, ss, 1);
    ss += __shfl_xor_sync(0xffffffffu, ss, 2);
    ss += __shfl_xor_sync(0xffffffffu, ss, 4);
    if (part == 0 && row0 + i * 32 < n_rows) {
      const float r = inv_or_zero(ss);
      if (r_f32 != nullptr) r_f32[row0 + i * 32] = r; else r_bf16[row0 + i * 32] = __float2bfloat16_rn(r);
    }
  }
}

__device__ __forceinline__ uint32_t mul_bf16x2(uint32_t a, uint32_t b) {
  const __nv_bfloat162 p = __hmul2(*reinterpret_cast<const __nv_bfloat162*>(&a), *reinterpret_cast<const __nv_bfloat162*>(&b));
  return *reinterpret_cast<const uint32_t*>(&p);
}
__device__ __forceinline__ uint4 lds128(uint32_t addr) {
  uint4 v;
  asm volatile("ld.shared.v4.b32 {%0,%1,%2,%3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(addr) : "memory");
  return v;
}

// Registers: 640 threads x 96 at launch; the four warps that issue and copy give theirs to the builders
// (128 x 64 + 512 x 104 = 640 x 96).
template <int N> __device__ __forceinline__ void regs_release() { asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(N)); }
template <int N> __device__ __forceinline__ void regs_take() { asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(N)); }

struct AArgs {
  __nv_bfloat16* out;
  const float* r_f32;            // [BH][T]: 1 / ||k||^2 (pre-pass)
  const __nv_bfloat16* r_bf16;   // ... where r_f32 is null
  int* device_status;
  int Tlen;
  int d_v;
  int BH;
  int n_pairs;                   // blocks of 256 queries of a head
  int chunk_pairs;               // ... of a chunk (the quadratic form: n_pairs)
  int n_chunks;
  int first_state;               // first chunk that has a state before it
  int wide_out;                  // rows of the output are 32-byte aligned
  int by_chunk;                  // order of the items: the blocks of a chunk one after the other
  const unsigned short* z;       // [BH][n_chunks][state rows] bf16: Z before each chunk
};

// XR = exact key scales: the weights are r s^2 rounded to bf16 once, instead of s^2, r and their product.  Taken by the chunked
// form with a state handed in or out and with feature groups, whose outputs were 3 to 8 % further from the 64-bit result (2-norm)
// than on the kernels that answer the short calls of the same kinds (2.9e-3 there; 2.2e-3 to 2.4e-3 with exact scales).  One packed multiply
// and twice the reads of r per pair: 4 x 16 heads x 4096 tokens of the quadratic form 126 -> 136 us, where nothing calls for
// it; 2 x 16 x 3001 with the state 109 -> 111.
// SPLIT = a work item is 128 queries without a state: both halves hold the same query tile, half A takes the even and half B the
// odd key tiles, and the epilogue adds their [O | D] (the weights are polynomial: partial sums simply add).  For calls of few
// blocks; see tc_attend.
// R = runs of 8 features that a row may have.  G = feature groups of the blockwise map: a key tile holds KT = 128 / G keys, and the 128 score columns of a buffer
// hold, for each half of those keys, the G per-group score blocks Q_a K_a^T side by side (group a in columns [a KT/2,
// a KT/2 + KT/2) of the sub-buffer); the weight of a key is the sum over the groups of the squared scores.
// VC = value columns: 64, or 32 for rows of values of up to 32 entries, whose tiles have rows of 64 bytes (64B swizzle) and whose
// apply and state MMAs N = 32 + 16 instead of 64 + 16 (128 heads x 2048 tokens of 32 entries 66.0 -> 62.3 us).
template <int G, int R, bool XR, bool SPLIT, int VC>
__global__ void __launch_bounds__(NTHREADS, 1)
tc_attend_kernel(const __grid_constant__ CUtensorMap tmQ, const __grid_constant__ CUtensorMap tmK,
                 const __grid_constant__ CUtensorMap tmV, const __grid_constant__ CUtensorMap tmS, const AArgs args) {
  extern __shared__ unsigned char smem_raw[];
  unsigned char* base = reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  auto bar = [&](int i) { return reinterpret_cast<uint64_t*>(base + OFF_BAR) + i; };
  auto stage = [&](int s) { return base + OFF_ST + s * STAGE_BYTES; };
  __shared__ uint32_t tmem_base_s;
  __shared__ int abort_s;
  volatile int* abort_flag = &abort_s;

  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  constexpr int KT = KTILE / G;                   // keys per tile
  constexpr int KH = KT / 2;                      // keys of a sub-tile
  constexpr int KPL = KT / 32;                    // keys per lane of the scale warp
  constexpr int NST = PairTable<G, R>::kSlices;      // state tiles
  constexpr uint32_t VROW = VC * 2;               // bytes of a row of a value or state tile
  // where the Z columns of a stage begin: 32 bytes of every row, for four stages (two, and the other two behind them)
  auto z_stage = [](uint32_t s) { return VC == 64 ? s * 32 : (s >> 1) * 16384 + (s & 1) * 32; };
  // byte offset of (row, 16-byte chunk) in such a tile, as TMA and the MMA descriptors swizzle it
  auto v_offset = [](uint32_t row, uint32_t chunk) { return VC == 64 ? sw128_offset(row, chunk) : row * 64u + ((chunk ^ ((row >> 1) & 3u)) << 4); };

  // Work items.  Rank -> (block of its chunk, chunk, head): the last blocks of the chunks (the most key tiles) first,
  // among them the chunks in descending order, so that chunk 0, which reads no state, comes last.  The n-th item of a CTA:
  // rounds of gridDim.x items, dealt forwards and backwards in turn, so that the CTA that got the heaviest item of one
  // round gets the lightest of the next.
  // With two dozen items per CTA and more (by_chunk) the blocks of a chunk follow one another instead, so that its state is
  // read from memory once and by the other blocks from L2; the deal keeps a CTA's share even (block p in one round, the
  // mirrored one in the next).  With fewer items the last round weighs more, and the two orders are level.  Heaviest first / by chunk,
  // us: 16 heads x 131072 tokens 2000 / 1890 on a cool chip and 2200 / 2070 in a long run, with two groups 1720 / 1620 and 1850 / 1760,
  // 64 x 16384 964 / 948, 32 x 32768 1009 / 1002, 128 x 8192 901 / 901; 16 x 32768 (14 items per CTA) 505 / 502, 128 x 4096 with two
  // groups 326 / 322.
  struct Item {
    int bh, chunk, q0;            // head, chunk, first query
    int k0;                       // first key tile (in tiles of KT keys)
    int nk_a, nk_b;               // key tiles of the halves (0: half B lies beyond the sequence)
    int ns;                       // state tiles (0: no state)
    int n_tiles;
  };
  const int per_block = args.n_chunks * args.BH;
  const int n_ranks = args.chunk_pairs * per_block;
  auto next_item = [&](int& n, Item& it) -> bool {   // the item at or after the n-th; n is left at it
    for (;; ++n) {
      const long long id = (long long)n * gridDim.x + ((n & 1) ? (int)gridDim.x - 1 - (int)blockIdx.x : (int)blockIdx.x);
      if ((long long)n * gridDim.x >= n_ranks) return false;
      if (id >= n_ranks) continue;
      int p, rem;
      if (args.by_chunk) {
        rem = (int)id / args.chunk_pairs;
        p = args.chunk_pairs - 1 - (int)id % args.chunk_pairs;
      } else {
        p = args.chunk_pairs - 1 - (int)id / per_block;
        rem = (int)id % per_block;
      }
      it.chunk = args.n_chunks - 1 - rem / args.BH;
      it.bh = rem % args.BH;
      const int pair = it.chunk * args.chunk_pairs + p;
      if (pair >= args.n_pairs) continue;
      if (SPLIT) {
        it.q0 = pair * QT;
        it.k0 = it.ns = 0;
        it.n_tiles = (p + 1) * G;
        it.nk_b = it.n_tiles / 2;
        it.nk_a = it.n_tiles - it.nk_b;
        return true;
      }
      it.q0 = pair * 2 * QT;
      it.k0 = it.chunk * args.chunk_pairs * 2 * G;
      it.nk_a = (2 * p + 1) * G;
      it.nk_b = it.q0 + QT < args.Tlen ? (2 * p + 2) * G : 0;
      it.ns = it.chunk >= args.first_state ? NST : 0;
      it.n_tiles = it.ns + (it.nk_b > 0 ? it.nk_b : it.nk_a);
      return true;
    }
  };

  if (tid == 0) {
    abort_s = 0;
    mbar_init(bar(BAR_QFULL), 1);
    mbar_init(bar(BAR_QEMPTY), 512);
    for (int i = 0; i < 2; ++i) {
      mbar_init(bar(BAR_QT + i), 128);
      mbar_init(bar(BAR_ODONE + i), 1);
      mbar_init(bar(BAR_OFREE + i), SPLIT ? 512 : 256);
    }
    for (int i = 0; i < 4; ++i) {
      mbar_init(bar(BAR_SFULL + i), 1);
      mbar_init(bar(BAR_PFULL + i), 128);
    }
    for (int i = 0; i < NSTAGE; ++i) {
      mbar_init(bar(BAR_FULL + i), 2);
      mbar_init(bar(BAR_EMPTY + i), 2);
    }
    for (int i = 0; i < 8; ++i) {
      mbar_init(bar(BAR_FFULL + i), 128);
      mbar_init(bar(BAR_SFREE + i), 1);
    }
    mbar_init(bar(BAR_DRAIN), 2);
    fence_mbar_init();
    tma_prefetch_desc(&tmQ);
    tma_prefetch_desc(&tmK);
    tma_prefetch_desc(&tmV);
    if (args.first_state < args.n_chunks) tma_prefetch_desc(&tmS);
  }
  // columns 64..127 of 16 rows of the value operand: [1, 0, ...] (every step of 16 rows reads the same block: the
  // descriptor's leading offset is the distance to it); the Z columns of the state start as zeros
  if (tid < VC * 2)
    *reinterpret_cast<uint4*>(base + OFF_ONES + v_offset(tid / (VC / 8), tid % (VC / 8))) = make_uint4(tid % (VC / 8) == 0 ? 0x3F80u : 0u, 0u, 0u, 0u);
  if (args.first_state < args.n_chunks)
    for (int i = tid; i < 2048; i += NTHREADS) *reinterpret_cast<uint4*>(base + OFF_Z + i * 16) = make_uint4(0u, 0u, 0u, 0u);
  fence_async_smem();
  if (warp == 0) {
    tmem_alloc(&tmem_base_s, TMEM_COLS);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tb = tmem_base_s;
  bool ok = true;
  // A programmatic dependent launch behind the state kernel, which may run for long: everybody waits for it here, where no
  // limit on time applies.  (Without states only warp 3 waits, for the key scales.)
  if (args.first_state < args.n_chunks) cudaGridDependencySynchronize();

  if (warp == 0) {
    regs_release<64>();
    // =========================== TMA producer ===========================
    if (elect_one()) {
      uint32_t it = 0;                                   // tiles loaded so far, over all items
      int ni = 0;
      Item w;
      for (int n = 0; ok && next_item(n, w); ++n, ++ni) {
        ok = wait_or_abort(bar(BAR_QEMPTY), (ni & 1) ^ 1, abort_flag);
        if (!ok) break;
        const bool two = !SPLIT && w.nk_b > 0;           // query tiles
        mbar_arrive_expect_tx(bar(BAR_QFULL), two ? 32768 : 16384);
        tma_load_3d(base + OFF_Q, &tmQ, bar(BAR_QFULL), 0, w.q0, w.bh);
        if (two) tma_load_3d(base + OFF_Q + 16384, &tmQ, bar(BAR_QFULL), 0, w.q0 + QT, w.bh);
        for (int j = 0; j < w.n_tiles && ok; ++j, ++it) {
          const int s = it % NSTAGE;
          ok = wait_or_abort(bar(BAR_EMPTY + s), ((it / NSTAGE) & 1) ^ 1, abort_flag);
          if (!ok) break;
          if (j >= w.ns) {
            const int key = (w.k0 + j - w.ns) * KT;
            mbar_arrive_expect_tx(bar(BAR_FULL + s), KT * (128 + VROW));   // K and V tiles
            tma_load_3d(stage(s), &tmK, bar(BAR_FULL + s), 0, key, w.bh);
            tma_load_3d(stage(s) + 16384, &tmV, bar(BAR_FULL + s), 0, key, w.bh);
          } else {
            const int slot = w.bh * args.n_chunks + w.chunk;
            mbar_arrive_expect_tx(bar(BAR_FULL + s), 256 * VROW);
            tma_load_3d(stage(s), &tmS, bar(BAR_FULL + s), 0, j * 256, slot);
          }
        }
      }
    }
  } else if (warp == 1 || warp == 2) {
    regs_release<64>();
    // =========================== MMA issuer of half A or B ===========================
    // The 128 columns of a half's buffer are two sub-buffers of 64, each a chain of its own.  Key tiles: open (score MMAs)
    // -> builders -> close (apply MMAs) -> open of the next tile; the thread goes round close 0, open 0, close 1, open 1,
    // so the chains run half a period apart.  State tiles: a sub-buffer is two pieces of 32 columns (64 features), which the
    // builders fill as they become free.  MMAs that overwrite columns follow the MMAs that read them in the same thread.
    if (elect_one()) {
      const int h = warp - 1;
      const uint32_t id_s = instr_desc(kFmtBF16, kFmtBF16, 0, 0, 128, KH);      // scores: B K-major
      const uint32_t id_p = instr_desc(kFmtBF16, kFmtBF16, 0, 1, 128, VC + 16); // apply, Psi(Q) [S | Z]: B MN-major, N = VC + 16
      const uint64_t dk = smem_desc(0, 16, 1024, kSwizzle128B);
      const uint32_t tS = tb + COL_S + h * 128, tO = tb + COL_O + h * 80, tQ = tb + COL_Q + h * 32;
      const uint32_t ones = smem_u32(base + OFF_ONES), zcol = smem_u32(base + OFF_Z);
      // MN-major: 8 rows of VROW bytes per atom (SBO), columns VC.. in the constant block (LBO)
      auto bdesc = [&](uint32_t addr, uint32_t extra) { return smem_desc(addr, extra - addr, 8 * VROW, VC == 64 ? kSwizzle128B : kSwizzle64B); };
      // ... moved by a number of bytes: the start address goes up and the distance to the constant block down
      auto move = [](uint64_t desc, uint32_t bytes) { return desc + (uint64_t)(bytes >> 4) * (1ull - (1ull << 16)); };
      const uint64_t dv0 = bdesc(smem_u32(stage(0)) + 16384, ones), dk0 = at(dk, smem_u32(stage(0)));
      uint32_t it = 0, cnt = 0, n_st = 0;   // tiles, key tiles of this half, its state tiles
      int n_done = 0;                       // items of this half so far
      Item w;
      for (int n = 0; ok && next_item(n, w); ++n) {
        const int nk = h == 0 ? w.nk_a : w.nk_b;
        const int nt = nk > 0 ? w.ns + nk : 0;      // tiles of this half
        uint32_t acc = 0;
        auto landed = [&](uint32_t g_it) { return wait_or_abort(bar(BAR_FULL + g_it % NSTAGE), (g_it / NSTAGE) & 1, abort_flag); };
        auto o_free = [&]() { return n_done == 0 || wait_or_abort(bar(BAR_OFREE + h), (n_done - 1) & 1, abort_flag); };
        auto open = [&](uint32_t g_it, int c) {
          const uint64_t d = dk0 + ((g_it % NSTAGE) * STAGE_BYTES + c * KH * 128) / 16;
#pragma unroll
          for (int ks = 0; ks < R / 2; ++ks)   // 16 features per step; group ks / (4 / G) accumulates over its own steps
            mma_f16_ts(tS + c * 64 + (ks / (4 / G)) * KH, tQ + ks * 8, d + ks * 2, id_s, (ks % (4 / G)) > 0);
          mma_commit(bar(BAR_SFULL + 2 * h + c));
        };
        auto close = [&](uint32_t g_it, int c) -> bool {
          if (!wait_or_abort(bar(BAR_PFULL + 2 * h + c), cnt & 1, abort_flag)) return false;
          tc_fence_after();
          const uint64_t d = move(dv0, (g_it % NSTAGE) * STAGE_BYTES + c * KH * VROW);
#pragma unroll
          for (int ks = 0; ks < KH / 16; ++ks) mma_f16_ts(tO, tS + c * 64 + ks * 8, move(d, ks * 16 * VROW), id_p, ks > 0 ? 1u : acc);
          acc = 1;
          return true;
        };
        if constexpr (SPLIT) {
          // every other tile is this half's; the others are passed on as they land (a parity cannot tell two phases of a
          // stage apart, so both halves see every tile)
          const uint32_t end = it + w.n_tiles;
          auto pass = [&](uint32_t g_it) -> bool {
            if (!landed(g_it)) return false;
            mbar_arrive(bar(BAR_EMPTY + g_it % NSTAGE));
            return true;
          };
          if (h == 1) ok = pass(it++);
          if (nk > 0) {
            ok = ok && wait_or_abort(bar(BAR_QT + h), n_done & 1, abort_flag) && landed(it);
            if (ok) {
              tc_fence_after();
              open(it, 0);
              open(it, 1);
              ok = o_free();
            }
            for (int j = 0; j < nk && ok; ++j, it += 2, ++cnt) {
              const bool next = j + 1 < nk;
              ok = (!next || (pass(it + 1) && landed(it + 2))) && close(it, 0);
              if (ok && next) open(it + 2, 0);
              ok = ok && close(it, 1);
              if (!ok) break;
              mma_commit(bar(BAR_EMPTY + it % NSTAGE));
              if (next) open(it + 2, 1);
              else if (it + 1 < end) ok = pass(it + 1);
            }
            if (ok) mma_commit(bar(BAR_ODONE + h));
            ++n_done;
          }
          it = end;
          continue;
        }
        if (nt > 0) ok = wait_or_abort(bar(BAR_QT + h), n_done & 1, abort_flag) && (w.ns > 0 || landed(it));
        if (nt > 0 && ok) {
          tc_fence_after();
          if (w.ns > 0) {
#pragma unroll 1
            for (int t = 0; t < NST && ok; ++t, ++it, ++n_st) {
              ok = landed(it) && (t > 0 || o_free()) && (t + 1 < NST || landed(it + 1));
              const uint64_t ds = bdesc(smem_u32(stage(it % NSTAGE)), zcol + z_stage(it % NSTAGE));
#pragma unroll
              for (int c = 0; c < 2; ++c) {
#pragma unroll
                for (int pp = 0; pp < 2; ++pp) {
                  ok = ok && wait_or_abort(bar(BAR_FFULL + 4 * h + 2 * c + pp), n_st & 1, abort_flag);
                  if (!ok) break;
                  tc_fence_after();
#pragma unroll
                  for (int ks = 0; ks < 4; ++ks)             // 16 rows at a time, of the state and of Z
                    mma_f16_ts(tO, tS + c * 64 + pp * 32 + ks * 8, ds + (c * 8 + pp * 4 + ks) * VROW, id_p, c + pp + ks > 0 ? 1u : acc);
                  acc = 1;
                  mma_commit(bar(BAR_SFREE + 4 * h + 2 * c + pp));
                }
                if (!ok) break;
                if (c == 1) mma_commit(bar(BAR_EMPTY + it % NSTAGE));
                if (t + 1 == NST) open(it + 1, c);       // the first key tile
              }
            }
          } else {
            open(it, 0);
            open(it, 1);
            ok = o_free();
          }
        }
        for (int j = 0; j < nk && ok; ++j, ++it, ++cnt) {
          const bool next = j + 1 < nk;
          ok = (!next || landed(it + 1)) && close(it, 0);
          if (ok && next) open(it + 1, 0);
          ok = ok && close(it, 1);
          if (!ok) break;
          mma_commit(bar(BAR_EMPTY + it % NSTAGE));
          if (next) open(it + 1, 1);
        }
        for (int j = nt; j < w.n_tiles && ok; ++j, ++it) {      // the other half's tiles
          ok = landed(it);
          if (ok) mbar_arrive(bar(BAR_EMPTY + it % NSTAGE));
        }
        if (nt > 0) {
          if (ok) mma_commit(bar(BAR_ODONE + h));
          ++n_done;
        }
      }
    }
  } else if (warp == 3) {
    regs_release<64>();
    // =========================== per tile: r = 1 / ||k||^2 of its keys, or its column of Z, to shared memory ===========================
    // (the key scale multiplies the weights, so the values are used as they are; a zero key row has r = 0: zero
    // feature).
    cudaGridDependencySynchronize();
    uint32_t it = 0;
    Item w;
    for (int n = 0; ok && next_item(n, w); ++n) {
      const size_t head = (size_t)w.bh * args.Tlen;
      const unsigned short* zs = args.z + ((size_t)w.bh * args.n_chunks + w.chunk) * (NST * 256);
      auto load = [&](int j, uint32_t (&x)[8]) {                  // tile j: r of KPL keys (fp32 or bf16), or Z of 8 rows (bf16), per lane
        if (j < w.ns) {
#pragma unroll
          for (int e = 0; e < 8; ++e) x[e] = zs[j * 256 + e * 32 + lane];
        } else {
#pragma unroll
          for (int e = 0; e < KPL; ++e) {
            const int key = (w.k0 + j - w.ns) * KT + lane * KPL + e;
            const bool in = j < w.n_tiles && key < args.Tlen;
            if (XR) x[e] = in ? __float_as_uint(args.r_f32[head + key]) : 0u;
            else if (args.r_f32 != nullptr) x[e] = in ? pack_bf16(args.r_f32[head + key], 0.f) : 0u;
            else x[e] = in ? reinterpret_cast<const unsigned short*>(args.r_bf16)[head + key] : 0u;
          }
        }
      };
      uint32_t x[8] = {};
      load(0, x);
      for (int j = 0; j < w.n_tiles && ok; ++j, ++it) {
        const int s = it % NSTAGE;
        uint32_t nx[8] = {};
        load(j + 1, nx);                // one tile ahead: the global-load latency stays off the ring
        ok = wait_or_abort(bar(BAR_EMPTY + s), ((it / NSTAGE) & 1) ^ 1, abort_flag);
        if (!ok) break;
        if (j < w.ns) {
#pragma unroll
          for (int e = 0; e < 8; ++e) {
            const int row = e * 32 + lane;
            const uint32_t z = VC == 64 ? v_offset(row, 2 * s) : (s >> 1) * 16384u + v_offset(row, 2 * (s & 1));
            *reinterpret_cast<unsigned short*>(base + OFF_Z + z) = (unsigned short)x[e];
          }
          fence_async_smem();
        } else {
#pragma unroll
          for (int e = 0; e < KPL; ++e) {
            if (XR) reinterpret_cast<uint32_t*>(base + OFF_RV + s * 512)[lane * KPL + e] = x[e];
            else reinterpret_cast<unsigned short*>(base + OFF_RV + s * 512)[lane * KPL + e] = (unsigned short)x[e];
          }
        }
#pragma unroll
        for (int e = 0; e < 8; ++e) x[e] = nx[e];
        __syncwarp();
        if (lane == 0) mbar_arrive(bar(BAR_FULL + s));      // (the builders of a key tile come after its score MMAs)
      }
    }
  } else {
    regs_take<104>();
    // =========================== builders (256 threads per half) ===========================
    const uint32_t q4 = warp & 3;
    const int bw = warp - WARP_BLD0;
    const int h = bw >> 3;                       // half
    const int ch = (bw >> 2) & 1;                // sub-buffer: the first or second half of the keys (features) of a tile
    const int rowl = q4 * 32 + lane;             // query row inside the tile (= TMEM lane)
    const uint32_t tS = tmem_addr(tb, q4 * 32, COL_S + h * 128 + ch * 64), tO = tmem_addr(tb, q4 * 32, COL_O + h * 80);
    const uint32_t qrow_s = smem_u32(base + OFF_Q) + (SPLIT ? 0 : h * 16384);
    // 16 bytes (eight features) of this thread's query row, from the item's tile in shared memory
    auto qrun = [&](int c) { return lds128(qrow_s + sw128_offset(rowl, c)); };
    // The query tile of an item into TMEM, by the warps of the second sub-buffer: the scores of an item's last tile are
    // issued sub-buffer 0 first, so only they know that no score MMA reads the tile of the item before any more.
    auto copy_q = [&](int ni, const Item& w) {
      ok = ok && wait_or_abort(bar(BAR_QFULL), ni & 1, abort_flag);
      if (!ok) return;
      if (ch == 1 && (h == 0 || w.nk_b > 0)) {
#pragma unroll
        for (int hf = 0; hf < 2; ++hf) {
          uint32_t r[16];
#pragma unroll
          for (int c = 0; c < 4; ++c) {
            const uint4 x = qrun(hf * 4 + c);
            r[4 * c] = x.x; r[4 * c + 1] = x.y; r[4 * c + 2] = x.z; r[4 * c + 3] = x.w;
          }
          tmem_st16(tmem_addr(tb, q4 * 32, COL_Q + h * 32 + hf * 16), r);
        }
        tmem_wait_st();
        tc_fence_before();
        mbar_arrive(bar(BAR_QT + h));
      }
      if (w.ns == 0) mbar_arrive(bar(BAR_QEMPTY));
    };
    uint32_t it = 0, cnt = 0, n_st = 0;
    int n_done = 0, ni = 0, n = 0;
    int n_done_b = 0;                            // SPLIT: items with tiles for half B (n_done: all)
    Item w;
    bool more = next_item(n, w);
    if (more) copy_q(0, w);
    for (; more && ok; ++ni) {
      const int nk = h == 0 ? w.nk_a : w.nk_b;
      const int qrow = w.q0 + (SPLIT ? 0 : h * QT) + rowl;
      const uint32_t it0 = it;
      it += w.n_tiles;
      if (nk > 0 && w.ns > 0) {
        // ---- the features of this query row, 256 per tile, this warp's two pairs of runs ----
        static constexpr PairTable<G, R> kPairs{};
#pragma unroll 1
        for (int t = 0; t < NST && ok; ++t, ++n_st) {
#pragma unroll 1
          for (int pp = 0; pp < 2; ++pp) {
            const int p = 4 * t + 2 * ch + pp;
            const uint4 xg = qrun(kPairs.g[p]), xh = qrun(kPairs.h[p]);
            const uint32_t gs[4] = {xg.x, xg.y, xg.z, xg.w}, hs[4] = {xh.x, xh.y, xh.z, xh.w};
            uint32_t f[32];
#pragma unroll
            for (int j = 0; j < 8; ++j) {
              const uint32_t b2 = (j & 1) ? __byte_perm(hs[j >> 1], 0, 0x3232) : __byte_perm(hs[j >> 1], 0, 0x1010);
#pragma unroll
              for (int e = 0; e < 4; ++e) f[4 * j + e] = mul_bf16x2(gs[e], b2);
            }
            // the piece is free: the item before is complete, or the MMAs of the tile before have read its features
            if (t > 0) ok = ok && wait_or_abort(bar(BAR_SFREE + 4 * h + 2 * ch + pp), (n_st - 1) & 1, abort_flag);
            if (!ok) break;
            tc_fence_after();
            tmem_st32(tS + pp * 32, f);
            tmem_wait_st();
            tc_fence_before();
            mbar_arrive(bar(BAR_FFULL + 4 * h + 2 * ch + pp));
          }
        }
        if (!ok) break;
      }
      if (w.ns > 0) mbar_arrive(bar(BAR_QEMPTY));
      for (int j = 0; j < nk && ok; ++j, ++cnt) {
        const int kj = SPLIT ? 2 * j + h : j;         // key tile of the item
        const uint32_t g_it = it0 + w.ns + kj;
        const int s = g_it % NSTAGE;
        ok = wait_or_abort(bar(BAR_SFULL + 2 * h + ch), cnt & 1, abort_flag);
        if (!ok) break;
        tc_fence_after();
        const bool diag = kj >= (SPLIT ? w.n_tiles : nk) - G;
        if constexpr (G > 1) {
          // this warp weighs keys [ch KT/2, ch KT/2 + KT/2) of the tile: one column run per group
          const int key0 = (w.k0 + kj) * KT + ch * KH;
          uint32_t y[G][KH], pk[KH / 2];
          const uint32_t rbase = smem_u32(base + OFF_RV) + s * 512 + ch * (KH * 4);   // fp32 r of this warp's keys, 4 per load
          const uint32_t* rw = reinterpret_cast<const uint32_t*>(base + OFF_RV + s * 512) + ch * (KH / 2);   // bf16 r, in pairs
#pragma unroll
          for (int g = 0; g < G; ++g) {
            if constexpr (KH == 32) tmem_ld32(tS + g * KH, y[g]); else tmem_ld16(tS + g * KH, y[g]);
          }
#pragma unroll
          for (int g = 0; g < G; ++g) tmem_wait_ld(y[g]);
          // two copies of the loop, chosen once per tile: the causal test exists on the diagonal tiles only
          auto weigh_g = [&](auto masked) {
#pragma unroll
            for (int c0 = 0; c0 < KH; c0 += 4) {
              uint4 t4 = make_uint4(0u, 0u, 0u, 0u);
              if (XR) t4 = lds128(rbase + c0 * 4);
              const float rr[4] = {__uint_as_float(t4.x), __uint_as_float(t4.y), __uint_as_float(t4.z), __uint_as_float(t4.w)};
#pragma unroll
              for (int c = c0; c < c0 + 4; c += 2) {
                float2 x = make_float2(0.f, 0.f);
#pragma unroll
                for (int g = 0; g < G; ++g) {
                  const float2 sv = make_float2(__uint_as_float(y[g][c]), __uint_as_float(y[g][c + 1]));
                  x = __ffma2_rn(sv, sv, x);
                }
                if (XR) x = __fmul2_rn(x, make_float2(rr[c - c0], rr[c - c0 + 1]));
                if constexpr (decltype(masked)::value) {
                  if (key0 + c > qrow) x.x = 0.f;
                  if (key0 + c + 1 > qrow) x.y = 0.f;
                }
                pk[c / 2] = XR ? pack_bf16(x.x, x.y) : mul_bf16x2(pack_bf16(x.x, x.y), rw[c / 2]);
              }
            }
          };
          if (diag) weigh_g(std::true_type{}); else weigh_g(std::false_type{});
          // the weights overwrite this warp's own score columns of group 0
          if constexpr (KH == 32) tmem_st16(tS, pk); else tmem_st8(tS, pk);
        } else {
          const uint32_t rbase = smem_u32(base + OFF_RV) + s * 512 + ch * (XR ? 256 : 128);   // r of this warp's 64 keys, 16 bytes per load
          const int key0 = (w.k0 + kj) * KT + ch * 64;
          // 32 columns at a time, each half behind a load of its own: a warp that runs through a hundred independent
          // instructions holds its scheduler, and the issuers, whose few instructions the MMAs wait for, get their slots when
          // it stalls (64 heads x 4096 tokens 124.1 -> 121.3 us; 16 columns at a time 123.4)
          auto weigh_tile = [&](auto masked) {
            constexpr int CW = 32, RPL = XR ? 4 : 8;             // columns at a time, keys per load of r
#pragma unroll
            for (int c0 = 0; c0 < 64; c0 += CW) {
              uint32_t y[CW], pk[CW / 2];
              tmem_ld32(tS + c0, y);
              tmem_wait_ld(y);
#pragma unroll
              for (int i = 0; i < CW / RPL; ++i) {
                const uint4 t4 = lds128(rbase + (c0 / RPL + i) * 16);
                const uint32_t rr[4] = {t4.x, t4.y, t4.z, t4.w};
#pragma unroll
                for (int e = 0; e < RPL; e += 2) {
                  const int jj = RPL * i + e;
                  const float2 sv = make_float2(__uint_as_float(y[jj]), __uint_as_float(y[jj + 1]));
                  float2 x = __fmul2_rn(sv, sv);
                  if constexpr (XR) x = __fmul2_rn(x, make_float2(__uint_as_float(rr[e]), __uint_as_float(rr[e + 1])));
                  if constexpr (decltype(masked)::value) {
                    if (key0 + c0 + jj > qrow) x.x = 0.f;
                    if (key0 + c0 + jj + 1 > qrow) x.y = 0.f;
                  }
                  pk[jj / 2] = XR ? pack_bf16(x.x, x.y) : mul_bf16x2(pack_bf16(x.x, x.y), rr[e / 2]);
                }
              }
              tmem_st16(tS + c0 / 2, pk);          // over scores that are in this warp's registers
            }
          };
          if (diag) weigh_tile(std::true_type{}); else weigh_tile(std::false_type{});
        }
        tmem_wait_st();
        tc_fence_before();
        mbar_arrive(bar(BAR_PFULL + 2 * h + ch));
      }
      if (!ok) break;
      // the next item's queries go to TMEM before the wait for this item's last MMAs
      const int bh = w.bh;
      const bool with_b = w.nk_b > 0;
      ++n;
      more = next_item(n, w);
      if (more) copy_q(ni + 1, w);
      if constexpr (SPLIT) {
        // ---- epilogue: the halves' [O | D] of these queries added, 16 columns per thread ----
        const uint32_t oa = tmem_addr(tb, q4 * 32, COL_O), c16 = (2 * h + ch) * 16;
        ok = ok && wait_or_abort(bar(BAR_ODONE), n_done & 1, abort_flag) &&
             (!with_b || wait_or_abort(bar(BAR_ODONE + 1), n_done_b & 1, abort_flag));
        if (!ok) break;
        ++n_done;
        n_done_b += with_b ? 1 : 0;
        tc_fence_after();
        uint32_t x[16], y[16], dx[4], dy[4];
        tmem_ld16(oa + c16, x);
        tmem_ld4(oa + VC, dx);
        tmem_ld16(oa + 80 + c16, y);
        tmem_ld4(oa + 80 + VC, dy);
        tmem_wait_ld(x);
        tmem_wait_ld(y);
        tmem_wait_ld(dx);
        tmem_wait_ld(dy);
        tc_fence_before();
        mbar_arrive(bar(BAR_OFREE));
        if (with_b) mbar_arrive(bar(BAR_OFREE + 1));
        const float den = __uint_as_float(dx[0]) + (with_b ? __uint_as_float(dy[0]) : 0.f);
        const float inv = den > 0.f ? 1.f / den : 0.f;
        if (qrow < args.Tlen) {
          __nv_bfloat16* dst = args.out + ((size_t)bh * args.Tlen + qrow) * args.d_v + c16;
          auto sum = [&](int c) { return (__uint_as_float(x[c]) + (with_b ? __uint_as_float(y[c]) : 0.f)) * inv; };
          uint4 pkt[2];
#pragma unroll
          for (int jj = 0; jj < 16; jj += 8)
            pkt[jj / 8] = make_uint4(pack_bf16(sum(jj), sum(jj + 1)), pack_bf16(sum(jj + 2), sum(jj + 3)),
                                     pack_bf16(sum(jj + 4), sum(jj + 5)), pack_bf16(sum(jj + 6), sum(jj + 7)));
          if ((int)c16 < args.d_v) store_32(dst, pkt, args.wide_out);          // (d_v is a multiple of 16)
        }
        continue;
      }
      if (nk == 0) continue;
      // ---- epilogue: out = O / D ----
      ok = ok && wait_or_abort(bar(BAR_ODONE + h), n_done & 1, abort_flag);
      if (!ok) break;
      ++n_done;
      tc_fence_after();
      uint32_t o[32], dn[4];
      tmem_ld32(tO + ch * 32, o);
      tmem_ld4(tO + VC, dn);
      tmem_wait_ld(o);
      tmem_wait_ld(dn);
      tc_fence_before();
      mbar_arrive(bar(BAR_OFREE + h));           // the MMAs of the next item may overwrite [O | D]
      const float den = __uint_as_float(dn[0]);
      const float inv = den > 0.f ? 1.f / den : 0.f;
      if (qrow < args.Tlen) {
        __nv_bfloat16* dst = args.out + ((size_t)bh * args.Tlen + qrow) * args.d_v + ch * 32;
#pragma unroll
        for (int jj = 0; jj < 32; jj += 16) {
          if (ch * 32 + jj >= args.d_v) break;
          uint4 pkt[2];
#pragma unroll
          for (int e = 0; e < 2; ++e) {
            const uint32_t* x = o + jj + 8 * e;
            pkt[e].x = pack_bf16(__uint_as_float(x[0]) * inv, __uint_as_float(x[1]) * inv);
            pkt[e].y = pack_bf16(__uint_as_float(x[2]) * inv, __uint_as_float(x[3]) * inv);
            pkt[e].z = pack_bf16(__uint_as_float(x[4]) * inv, __uint_as_float(x[5]) * inv);
            pkt[e].w = pack_bf16(__uint_as_float(x[6]) * inv, __uint_as_float(x[7]) * inv);
          }
          store_32(dst + jj, pkt, args.wide_out);      // (by sixteens 64 heads x 4096 tokens took 148.6 instead of 146.7 us)
        }
      }
    }
  }

  // ---------------- teardown ----------------
  if (!ok && args.device_status != nullptr) atomicExch(args.device_status, (int)KATA_ERR_DEVICE_TIMEOUT);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  if ((warp == 1 || warp == 2) && elect_one()) {
    mma_commit(bar(BAR_DRAIN));
    mbar_wait(bar(BAR_DRAIN), 0);
  }
  __syncthreads();
  if (warp == 0) tmem_dealloc(tb, TMEM_COLS);
}

}  // namespace

// workspace: r [BH][T] bf16
size_t tc_quadratic_workspace_bytes(const Problem& p) { return ((size_t)p.B * p.H * p.T * 2 + 255) / 256 * 256; }

void tc_rscale(const Problem& p, const KeyScales& r, LaunchCtx& ctx) {
  const size_t n_rows = (size_t)p.B * p.H * p.T;
  rscale_kernel<<<(unsigned)((n_rows + 32 * RS_ROWS - 1) / (32 * RS_ROWS)), 256, 0, ctx.stream>>>(static_cast<const __nv_bfloat16*>(p.k), r.f32,
                                                                                                          r.bf16, n_rows, p.d_k);
  note_launch(ctx);
}

void tc_attend(const Problem& p, const KeyScales& r, const AttendStates& st, int* device_status, LaunchCtx& ctx) {
  const int BH = p.B * p.H;
  CUtensorMap tmQ, tmK, tmV, tmS;
  const int kt = KTILE / p.groups;
  const bool narrow = tc_narrow(p);
  const int vc = narrow && p.d_v <= 32 ? 32 : 64;
  // No states and not more blocks of 256 queries than SMs: the call lasts as long as its longest block, so the halves of a CTA
  // share out the keys of one block of 128 queries instead (SPLIT).  From four tiles of the longest half on; shorter ones gain
  // nothing, and with more blocks the tiles that only one half uses cost more than the finer deal gives (with feature groups,
  // whose tiles cost more weighing per byte, the line lies a third higher).  Measured, us, blocks of 256 / split:
  //   one head x 8192 48 / 35, with two groups 87 / 52, with four 149 / 86; 6 x 4096 (96 blocks) 31.1 / 22.9, 8 x 4096 (128)
  //   31.3 / 24.3, 24 x 1500 (144) 18.2 / 16.4, 37 x 1024 (148) 14.7 / 14.4; 12 x 4096 (192) 31.9 / 33.8, 64 x 4096 130 / 181
  //   two groups 12 x 4096 (192) 50.8 / 45.2, 37 x 1500 (222) 24.6 / 26.7; four groups 81.9 / 70.3, 36.2 / 36.9
  //   short: 64 x 512 12.3 / 12.3
  const int n_blocks = (p.T + 2 * QT - 1) / (2 * QT);
  const bool split = st.n_chunks == 0 && n_blocks >= 2 && n_blocks * p.groups >= 4 && 3LL * BH * n_blocks <= (p.groups > 1 ? 4 : 3) * sm_count();
  const int n_pairs = split ? (p.T + QT - 1) / QT : n_blocks;
  AArgs a{static_cast<__nv_bfloat16*>(p.out), r.f32, r.bf16, device_status, p.T, p.d_v, BH, n_pairs, n_pairs, 1, 1, (reinterpret_cast<uintptr_t>(p.out) & 31) == 0, 0, nullptr};
  bool maps = make_tile_map(&tmQ, p.q, BH, p.T, QT, p.d_k) && make_tile_map(&tmK, p.k, BH, p.T, kt, p.d_k) &&
              make_tile_map(&tmV, p.v, BH, p.T, kt, p.d_v, vc);
  if (st.n_chunks > 0) {
    a.chunk_pairs = st.chunk_tokens / (2 * QT);
    a.n_chunks = st.n_chunks;
    a.first_state = st.first_state;
    a.by_chunk = (long long)BH * st.n_chunks * a.chunk_pairs >= 24LL * sm_count() ? 1 : 0;
    a.z = reinterpret_cast<const unsigned short*>(st.z);
    maps = maps && make_tile_map(&tmS, st.s, BH * st.n_chunks, tc_state_rows(p), 256, 64, vc);
  } else {
    tmS = tmK;
  }
  if (!maps) {
    ctx.status = KATA_ERR_CUDA;
    return;
  }
  void (*kern)(CUtensorMap, CUtensorMap, CUtensorMap, CUtensorMap, AArgs) = nullptr;
  auto pick = [&](auto g, auto r, auto xr, auto cols) {
    constexpr auto K = tc_attend_kernel<decltype(g)::value, decltype(r)::value, decltype(xr)::value, false, decltype(cols)::value>;
    constexpr auto KS = tc_attend_kernel<decltype(g)::value, decltype(r)::value, decltype(xr)::value, true, decltype(cols)::value>;
    kern = split ? KS : K;
    return split ? allow_smem<KS>((int)SMEM_ALLOC) : allow_smem<K>((int)SMEM_ALLOC);
  };
  using std::integral_constant;
  auto pick_g = [&](auto xr) {
    constexpr integral_constant<int, 64> c64{};
    if (p.groups == 2) return pick(integral_constant<int, 2>{}, integral_constant<int, 8>{}, xr, c64);
    if (p.groups == 4) return pick(integral_constant<int, 4>{}, integral_constant<int, 8>{}, xr, c64);
    return pick(integral_constant<int, 1>{}, integral_constant<int, 8>{}, xr, c64);
  };
  if (!(vc == 32            ? pick(integral_constant<int, 1>{}, integral_constant<int, 4>{}, std::false_type{}, integral_constant<int, 32>{})
        : narrow            ? pick(integral_constant<int, 1>{}, integral_constant<int, 4>{}, std::false_type{}, integral_constant<int, 64>{})
        : st.exact_scales   ? pick_g(std::true_type{})
                            : pick_g(std::false_type{}))) {
    ctx.status = KATA_ERR_CUDA;
    return;
  }
  const int sms = sm_count();
  const long long n_items = (long long)BH * n_pairs;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(n_items < sms ? n_items : sms));   // persistent: one CTA per SM
  cfg.blockDim = dim3(NTHREADS);
  cfg.dynamicSmemBytes = SMEM_ALLOC;
  cfg.stream = ctx.stream;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  if (cudaLaunchKernelEx(&cfg, kern, tmQ, tmK, tmV, tmS, a) != cudaSuccess) {
    cudaGetLastError();
    ctx.status = KATA_ERR_CUDA;
    return;
  }
  ++ctx.launches;
}

void tc_quadratic(const Problem& p, void* workspace, int* device_status, LaunchCtx& ctx) {
  const KeyScales r{nullptr, static_cast<__nv_bfloat16*>(workspace)};
  tc_rscale(p, r, ctx);
  if (ctx.status == KATA_OK) tc_attend(p, r, AttendStates{}, device_status, ctx);
}

}  // namespace kata
