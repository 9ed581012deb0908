// Chunk states of the chunked KATA forward on the Blackwell tensor cores (tcgen05 + TMEM), bf16:
//   S_[c+1] = S_[c] + Psi(K_[c])^T V_[c],  Z_[c+1] = Z_[c] + Psi(K_[c])^T 1     (section "Chunkwise forward")
// for chunks of a few hundred tokens, written out once per chunk for the attend kernel (kata_tc_attend.cu).
//
// One CTA = one head x one slice of 256 of the packed state rows (four block pairs, kata_pairs.cuh) x one segment of the
// chunk axis.  It walks tiles of 128 tokens:
//   operand  A[f, t] = (r_t k_t,b) k_t,a   features on the TMEM lanes, tokens on the columns.  A builder warp takes the
//            key tile in MMA-fragment form, transposed on the way (ldmatrix.trans: lane = (feature of a run of 8, pair of
//            tokens)), multiplies the fragment of run h by the key scales (r as the sum of two bf16, so that r k_b is rounded
//            once and a feature twice: with r rounded first the exported state was 2.9e-3 off in the 2-norm instead of
//            2.35e-3), leaves it in a scratch of its own from which
//            each of its features b is broadcast to the lanes (16 bytes = 4 runs of tokens per load), and multiplies the
//            fragments of the runs g by it.  tcgen05.st.16x128b takes exactly this layout, so the operand never passes
//            through shared memory.
//   update   [S | Z] += A [V | 1]   A from TMEM, B = the value tile as it is and a constant column of ones, N = 80,
//            two accumulators of 128 rows
// The accumulators carry the sum over all chunks so far (fp32); between chunks eight warps copy them out, one state row per
// thread: the state before the next chunk in bf16, pair weights included.  The builders run up to five half tiles ahead, so
// the MMAs that wait for the copy catch up.
//
// What bounds it.  Per tile and CTA 640 cycles of MMA, and about 1600 at present: the load/store pipe delivers 128 bytes a cycle
// to registers, and the builders' fragments (192), key scales (128), scaled runs (64) and broadcasts (270) take some 760 cycles
// of it, beside 256 for the TMA writes and 320 for the value operand on the shared memory.  The states leave by TMA from
// staging rows: stored by the copy warps, 16 bytes of a row per lane, they were another 344 cycles of that pipe per tile (16
// heads x 32768: 446 k cycles of the kernel, 392 k now; 131072 2.20 -> 2.00 ms a call).  Built in shared memory and read by the
// MMAs from there, as products of token rows, the A operand alone took 1024.  A builder warp takes about 1300 cycles for a half
// tile, most of it latency, so four sets of four take turns (two sets: 1460 cycles a tile of the kernel of that time).
//
// When the heads alone do not fill the GPU the chunk axis is cut into segments: every segment sums from zero and writes
// fp32, and state_fix_kernel adds the segments before it and rounds.
//
// Warps (896 threads): 0 TMA producer, 1 MMA issuer, 2 key scales, 4-19 builders (quadrant = warp % 4, four sets taking
// every fourth half tile), 20-27 copies.  All waits are bounded.
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
constexpr int CT = 128;          // tokens per tile
constexpr int NSTAGE = 4;
constexpr int NSLOT = 5;         // A operand: slots of 64 tokens x 256 features
constexpr int NSET = 4;          // sets of builder warps
constexpr int NTHREADS = 896;
constexpr int WARP_BLD0 = 4, WARP_CPY0 = 20;

constexpr uint32_t COL_ACC = 0;          // 2 (tiles of 128 rows) x 80
constexpr uint32_t COL_A = 160;          // NSLOT x 2 x 32
constexpr uint32_t TMEM_COLS = 512;

constexpr uint32_t STAGE_BYTES = 32768;                     // key tile, value tile
constexpr uint32_t OFF_ONES = NSTAGE * STAGE_BYTES;         // 16 rows of [1, 0 ...]: columns 64.. of the values
constexpr uint32_t OFF_RV = OFF_ONES + 2048;                // NSTAGE x 2 x 128 bf16 key scales (high and low parts), in the builders' order
constexpr uint32_t OFF_SCR = OFF_RV + NSTAGE * 512;         // 16 builder warps x 2 KB: scaled fragments of run h
constexpr uint32_t OFF_OUT = OFF_SCR + 16 * 2048;           // 8 copy warps x 32 state rows of 128 bytes, 128B swizzle
constexpr uint32_t OFF_BAR = OFF_OUT + 8 * 4096;
static_assert(OFF_OUT % 1024 == 0, "swizzle");
constexpr uint32_t SMEM_BYTES = OFF_BAR + 256;
constexpr uint32_t SMEM_ALLOC = SMEM_BYTES + 1024;
static_assert(SMEM_ALLOC > 116 * 1024, "one CTA per SM is assumed (the CTA allocates all of TMEM)");

enum {
  BAR_FULL = 0,      // [NSTAGE] tiles (TMA bytes) and their key scales (scale warp) landed
  BAR_EMPTY = 4,     // [NSTAGE] stage free: eight builder warps and the issuer's commit
  BAR_AFULL = 8,     // [NSLOT] operand slot built (four warps)
  BAR_AEMPTY = 13,   // [NSLOT] ... and consumed
  BAR_CFULL = 18,    // the MMAs of a chunk are complete
  BAR_CFREE = 19,    // the accumulators have been read, or set to the state handed in (256)
  BAR_DRAIN = 20,
  BAR_COUNT = 21
};

struct SArgs {
  const float* rscale;           // [BH][T]
  __nv_bfloat16* s;              // [BH][n_chunks][rows][64]: state before each chunk (one segment)
  __nv_bfloat16* z;              // [BH][n_chunks][rows]
  float* s_loc;                  // [BH][n_chunks][rows][64]: sum of the segment up to and including the chunk (several segments)
  float* z_loc;                  // [BH][n_chunks][rows]
  const float* s_init;           // state before the first token, public layout (null: zero)
  const float* z_init;
  float* s_final;                // state after the last token, public layout (null: not wanted); one segment only
  float* z_final;
  int wide_final;                // s_final is 32-byte aligned
  int packed;                    // public layout: packed upper triangles instead of direct
  int* device_status;
  int Tlen;
  int chunk_tiles, n_chunks;
  int walk_chunks;               // chunks whose sums are needed: n_chunks, or one less
  int seg_chunks;                // chunks per segment
};

// Row of the public state layout for the pair of features (a, b), a <= b, of the map with G blocks; direct: row (a, b).
template <int G> __device__ __forceinline__ int public_row(int a, int b, int packed) {
  constexpr int m = D / G;
  const int blk = a / m;
  a -= blk * m;
  b -= blk * m;
  return packed ? blk * (m * (m + 1) / 2) + a * m - a * (a - 1) / 2 + (b - a) : blk * m * m + a * m + b;
}
template <int G> __device__ __forceinline__ size_t public_rows(int packed) {
  constexpr int m = D / G;
  return packed ? (size_t)G * m * (m + 1) / 2 : (size_t)G * m * m;
}

template <int N> __device__ __forceinline__ void regs_release() { asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(N)); }
template <int N> __device__ __forceinline__ void regs_take() { asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(N)); }
static_assert(128 * 40 + 512 * 80 + 256 * 72 <= 896 * 72, "register budget");

__device__ __forceinline__ uint32_t mul_bf16x2(uint32_t a, uint32_t b) {
  const __nv_bfloat162 p = __hmul2(*reinterpret_cast<const __nv_bfloat162*>(&a), *reinterpret_cast<const __nv_bfloat162*>(&b));
  return *reinterpret_cast<const uint32_t*>(&p);
}
// x (hi + lo), rounded once (the rounding of the small term does not count)
__device__ __forceinline__ uint32_t scale_bf16x2(uint32_t x, uint32_t hi, uint32_t lo) {
  const uint32_t low = mul_bf16x2(x, lo);
  const __nv_bfloat162 p = __hfma2(*reinterpret_cast<const __nv_bfloat162*>(&x), *reinterpret_cast<const __nv_bfloat162*>(&hi),
                                   *reinterpret_cast<const __nv_bfloat162*>(&low));
  return *reinterpret_cast<const uint32_t*>(&p);
}
// Four 8 x 8 blocks, each transposed: lane i gets column i / 4, rows 2 (i % 4) and 2 (i % 4) + 1, of block j in r[j].
__device__ __forceinline__ void ldmatrix_x4_trans(uint32_t (&r)[4], uint32_t saddr) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(saddr) : "memory");
}
// 16 lanes x 32 columns: thread i holds row i / 4 (even registers) and i / 4 + 8 (odd), column 4 k + i % 4 in r[2k], r[2k+1].
__device__ __forceinline__ void tmem_st_16x128b_x8(uint32_t taddr, const uint32_t (&r)[16]) {
  asm volatile("tcgen05.st.sync.aligned.16x128b.x8.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16};"
               ::"r"(taddr), "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]), "r"(r[8]),
               "r"(r[9]), "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15]) : "memory");
}
__device__ __forceinline__ void lds128(uint32_t (&r)[4], uint32_t addr) {
  asm volatile("ld.shared.v4.b32 {%0,%1,%2,%3}, [%4];" : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr) : "memory");
}
__device__ __forceinline__ void sts128(uint32_t addr, const uint32_t (&r)[4]) {
  asm volatile("st.shared.v4.b32 [%0], {%1,%2,%3,%4};" ::"r"(addr), "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]) : "memory");
}

__device__ __forceinline__ void st_global_v8(float* p, const float4& a, const float4& b) {      // 32-byte aligned
  asm volatile("st.global.v8.f32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8};"
               ::"l"(p), "f"(a.x), "f"(a.y), "f"(a.z), "f"(a.w), "f"(b.x), "f"(b.y), "f"(b.z), "f"(b.w) : "memory");
}

template <int G, int R>
__global__ void __launch_bounds__(NTHREADS, 1)
tc_state_kernel(const __grid_constant__ CUtensorMap tmK, const __grid_constant__ CUtensorMap tmV, const __grid_constant__ CUtensorMap tmOut,
                const SArgs args) {
  extern __shared__ unsigned char smem_raw[];
  unsigned char* base = reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  auto bar = [&](int i) { return reinterpret_cast<uint64_t*>(base + OFF_BAR) + i; };
  auto stage = [&](int s) { return base + s * STAGE_BYTES; };
  __shared__ uint32_t tmem_base_s;
  __shared__ int abort_s;
  volatile int* abort_flag = &abort_s;
  static constexpr PairTable<G, R> kPairs{};
  constexpr int ROWS = PairTable<G, R>::kRows;

  cudaTriggerProgrammaticLaunchCompletion();      // the kernel behind starts on the SMs that this one leaves
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int slice = blockIdx.x, bh = blockIdx.y;
  const int c_beg = blockIdx.z * args.seg_chunks, c_end = min(c_beg + args.seg_chunks, args.walk_chunks);
  const int n_tiles_all = (args.Tlen + CT - 1) / CT;
  const int t_beg = c_beg * args.chunk_tiles, t_end = min(c_end * args.chunk_tiles, n_tiles_all);
  const int n = t_end - t_beg;                    // tiles of this CTA
  const bool first = c_beg == 0 && args.s_init != nullptr;      // starts from the state handed in

  if (tid == 0) {
    abort_s = 0;
    for (int i = 0; i < NSTAGE; ++i) {
      mbar_init(bar(BAR_FULL + i), 2);
      mbar_init(bar(BAR_EMPTY + i), 9);        // eight warps of the two sets that read a tile, and the MMAs
    }
    for (int i = 0; i < NSLOT; ++i) {
      mbar_init(bar(BAR_AFULL + i), 4);
      mbar_init(bar(BAR_AEMPTY + i), 1);
    }
    mbar_init(bar(BAR_CFULL), 1);
    mbar_init(bar(BAR_CFREE), 256);
    mbar_init(bar(BAR_DRAIN), 1);
    fence_mbar_init();
    tma_prefetch_desc(&tmK);
    tma_prefetch_desc(&tmV);
  }
  if (tid < 128)
    *reinterpret_cast<uint4*>(base + OFF_ONES + sw128_offset(tid >> 3, tid & 7)) = make_uint4((tid & 7) == 0 ? 0x3F80u : 0u, 0u, 0u, 0u);
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

  if (warp == 0) {
    regs_release<40>();
    // =========================== TMA producer ===========================
    if (elect_one()) {
      for (int j = 0; j < n && ok; ++j) {
        const int s = j % NSTAGE;
        ok = wait_or_abort(bar(BAR_EMPTY + s), ((j / NSTAGE) & 1) ^ 1, abort_flag);
        if (!ok) break;
        mbar_arrive_expect_tx(bar(BAR_FULL + s), 32768);
        tma_load_3d(stage(s), &tmK, bar(BAR_FULL + s), 0, (t_beg + j) * CT, bh);
        tma_load_3d(stage(s) + 16384, &tmV, bar(BAR_FULL + s), 0, (t_beg + j) * CT, bh);
      }
    }
  } else if (warp == 1) {
    regs_release<40>();
    // =========================== update issuer ===========================
    if (elect_one()) {
      const uint32_t idesc = instr_desc(kFmtBF16, kFmtBF16, 0, 1, 128, 80);
      // 16 tokens per 2 KB; a step moves the start address up and the distance to the constant block down
      const uint32_t v0 = smem_u32(stage(0)) + 16384;
      const uint64_t dv = smem_desc(v0, smem_u32(base + OFF_ONES) - v0, 1024, kSwizzle128B);
      auto move = [](uint64_t desc, uint32_t bytes) { return desc + (uint64_t)(bytes >> 4) * (1ull - (1ull << 16)); };
      int chunk_i = 0, in_chunk = 0;     // chunk of this segment, tile inside it
      const int first_free = first ? 1 : 0;
      for (int j = 0; j < n && ok; ++j) {
        const int s = j % NSTAGE;
        ok = wait_or_abort(bar(BAR_FULL + s), (j / NSTAGE) & 1, abort_flag);
        if (ok && in_chunk == 0 && chunk_i + first_free >= 1)       // the accumulators have been copied out, or set
          ok = wait_or_abort(bar(BAR_CFREE), (chunk_i + first_free - 1) & 1, abort_flag);
        const uint64_t ds = move(dv, s * STAGE_BYTES);
        const uint32_t acc = first || j > 0 ? 1u : 0u;
#pragma unroll
        for (int th = 0; th < 2; ++th) {
          const int hs = 2 * j + th, slot = hs % NSLOT;
          ok = ok && wait_or_abort(bar(BAR_AFULL + slot), (hs / NSLOT) & 1, abort_flag);
          if (!ok) break;
          tc_fence_after();
#pragma unroll
          for (int m = 0; m < 2; ++m)
#pragma unroll
            for (int ks = 0; ks < 4; ++ks)
              mma_f16_ts(tb + COL_ACC + m * 80, tb + COL_A + slot * 64 + m * 32 + ks * 8, move(ds, (th * 4 + ks) * 2048), idesc,
                         th > 0 || ks > 0 ? 1u : acc);
          mma_commit(bar(BAR_AEMPTY + slot));
        }
        if (!ok) break;
        mma_commit(bar(BAR_EMPTY + s));
        if (++in_chunk == args.chunk_tiles || j + 1 == n) {
          mma_commit(bar(BAR_CFULL));
          in_chunk = 0;
          ++chunk_i;
        }
      }
    }
  } else if (warp == 2) {
    regs_release<40>();
    // =========================== key scales, from the pre-pass to shared memory ===========================
    cudaGridDependencySynchronize();
    const float* rs = args.rscale + (size_t)bh * args.Tlen;
    auto load_r = [&](int j, float (&w)[4]) {             // tokens 4 lane .. 4 lane + 3 of tile j
      const int t0 = (t_beg + j) * CT + 4 * lane;
#pragma unroll
      for (int e = 0; e < 4; ++e) w[e] = (j < n && t0 + e < args.Tlen) ? rs[t0 + e] : 0.f;
    };
    float w[4];
    load_r(0, w);
    for (int j = 0; j < n && ok; ++j) {
      const int s = j % NSTAGE;
      float nx[4];
      load_r(j + 1, nx);
      ok = wait_or_abort(bar(BAR_EMPTY + s), ((j / NSTAGE) & 1) ^ 1, abort_flag);
      if (!ok) break;
      // a builder lane wants the pairs i % 4 of four consecutive runs of eight tokens: word (i % 4) * 4 + run of a group of 32
#pragma unroll
      for (int e = 0; e < 2; ++e) {
        const int pr = 2 * lane + e, grp = pr >> 4, run = (pr >> 2) & 3, i4 = pr & 3;
        unsigned char* dst = base + OFF_RV + s * 512 + (grp * 16 + i4 * 4 + run) * 4;
        const uint32_t hi = pack_bf16(w[2 * e], w[2 * e + 1]);
        auto low = [](float x, float h) { return isinf(h) ? 0.f : x - h; };
        *reinterpret_cast<uint32_t*>(dst) = hi;
        *reinterpret_cast<uint32_t*>(dst + 256) =
            pack_bf16(low(w[2 * e], __uint_as_float(hi << 16)), low(w[2 * e + 1], __uint_as_float(hi & 0xFFFF0000u)));
        w[2 * e] = nx[2 * e];
        w[2 * e + 1] = nx[2 * e + 1];
      }
      __syncwarp();
      if (lane == 0) mbar_arrive(bar(BAR_FULL + s));
    }
  } else if (warp == 3) {
    regs_release<40>();
  } else if (warp < WARP_CPY0) {
    regs_take<80>();
    // =========================== builders ===========================
    const int q4 = warp & 3, set = (warp - WARP_BLD0) >> 2, th = set & 1;   // half of the tiles j with j % 2 = set / 2
    const int pa = 4 * slice + (q4 >> 1), pb = pa + 2;
    const int ga = kPairs.g[pa], gb = kPairs.g[pb], ha = kPairs.h[pa], hb = kPairs.h[pb];
    const uint32_t scr = smem_u32(base + OFF_SCR) + (warp - WARP_BLD0) * 2048, scr_w = scr + lane * 16;
    const uint32_t scr_b = scr + (q4 & 1) * 256 + (lane & 3) * 16;   // feature 8 h + 4 (q4 & 1), this lane's token pairs
    // lane i of an ldmatrix addresses token i of 32 (run i / 8): byte offsets of the three or four runs of features
    const uint32_t row_off = (uint32_t)(th * 64 + lane) * 128u, sw = (uint32_t)(lane & 7);
    const uint32_t o_ga = row_off + (((uint32_t)ga ^ sw) << 4), o_gb = row_off + (((uint32_t)gb ^ sw) << 4);
    const uint32_t o_ha = row_off + (((uint32_t)ha ^ sw) << 4), o_hb = row_off + (((uint32_t)hb ^ sw) << 4);
    // (two copies of the loop: the pairs share the run h or have one each)
    auto build = [&](auto two) {
      constexpr bool TWO = decltype(two)::value;
      for (int j = set >> 1; j < n && ok; j += NSET / 2) {
        const int s = j % NSTAGE, hs = 2 * j + th, slot = hs % NSLOT;
        ok = wait_or_abort(bar(BAR_FULL + s), (j / NSTAGE) & 1, abort_flag);
        if (!ok) break;
        const uint32_t kt = smem_u32(stage(s)), rv = smem_u32(base + OFF_RV) + s * 512 + th * 128 + (lane & 3) * 16;
        uint32_t fa[2][4], fb[2][4];
#pragma unroll
        for (int grp = 0; grp < 2; ++grp) {                    // 32 tokens
          uint32_t fh[4], fk[4], r4[4], l4[4];
          ldmatrix_x4_trans(fh, kt + o_ha + grp * 4096);
          if constexpr (TWO) ldmatrix_x4_trans(fk, kt + o_hb + grp * 4096);
          lds128(r4, rv + grp * 64);
          lds128(l4, rv + 256 + grp * 64);
          ldmatrix_x4_trans(fa[grp], kt + o_ga + grp * 4096);
          ldmatrix_x4_trans(fb[grp], kt + o_gb + grp * 4096);
#pragma unroll
          for (int o = 0; o < 4; ++o) fh[o] = scale_bf16x2(fh[o], r4[o], l4[o]);
          sts128(scr_w + grp * 512, fh);
          if constexpr (TWO) {
#pragma unroll
            for (int o = 0; o < 4; ++o) fk[o] = scale_bf16x2(fk[o], r4[o], l4[o]);
            sts128(scr_w + 1024 + grp * 512, fk);
          }
        }
        __syncwarp();
        ok = wait_or_abort(bar(BAR_AEMPTY + slot), ((hs / NSLOT) & 1) ^ 1, abort_flag);
        if (!ok) break;
        tc_fence_after();
        const uint32_t ta = tmem_addr(tb, q4 * 32, COL_A + slot * 64);
#pragma unroll
        for (int jp = 0; jp < 2; ++jp) {                       // features b of run h, two at a time (16 lanes)
          uint32_t xa[16], xb[16];
#pragma unroll
          for (int e = 0; e < 2; ++e)
#pragma unroll
            for (int grp = 0; grp < 2; ++grp) {
              uint32_t b[4], b2[4];
              lds128(b, scr_b + (2 * jp + e) * 64 + grp * 512);
              if constexpr (TWO) lds128(b2, scr_b + 1024 + (2 * jp + e) * 64 + grp * 512);
#pragma unroll
              for (int o = 0; o < 4; ++o) {
                xa[2 * (4 * grp + o) + e] = mul_bf16x2(fa[grp][o], b[o]);
                xb[2 * (4 * grp + o) + e] = mul_bf16x2(fb[grp][o], TWO ? b2[o] : b[o]);
              }
            }
          tmem_st_16x128b_x8(ta + ((uint32_t)(jp * 16) << 16), xa);
          tmem_st_16x128b_x8(ta + ((uint32_t)(jp * 16) << 16) + 32, xb);
        }
        tmem_wait_st();
        tc_fence_before();
        __syncwarp();                                          // (also before the scratch is written again)
        if (lane == 0) {
          mbar_arrive(bar(BAR_AFULL + slot));
          mbar_arrive(bar(BAR_EMPTY + s));                     // this warp's part of the key tile has been used
        }
      }
    };
    if (ha != hb) build(std::true_type{}); else build(std::false_type{});
  } else {
    // =========================== copies: one state row per thread ===========================
    const int q4 = warp & 3, m = (warp - WARP_CPY0) >> 2;
    const int row = slice * 256 + m * 128 + q4 * 32 + lane;
    const int p = 4 * slice + 2 * m + (q4 >> 1), e = (q4 & 1) * 32 + lane;
    const int a = 8 * kPairs.g[p] + (e & 7), b = 8 * kPairs.h[p] + (e >> 3);
    const bool mirror = kPairs.g[p] != kPairs.h[p];          // the pair also stands for (b, a)
    const float wgt = mirror ? 2.f : 1.f;
    const int prow = public_row<G>(min(a, b), max(a, b), args.packed);
    const size_t n_pub = public_rows<G>(args.packed);
    const uint32_t ta = tmem_addr(tb, q4 * 32, COL_ACC + m * 80);
    // bf16 state of chunk c, rows of this warp: columns [col, col + 32) from x into its staging rows, and with the second half
    // all of them out by one TMA store
    unsigned char* out_rows = base + OFF_OUT + (warp - WARP_CPY0) * 4096;
    auto put_state = [&](int c, int col, const float (&x)[32]) {
      if (col == 0) {
        if (lane == 0) bulk_wait_read();           // the store of the chunk before has read the rows
        __syncwarp();
      }
#pragma unroll
      for (int i = 0; i < 4; ++i)
        *reinterpret_cast<uint4*>(out_rows + sw128_offset(lane, col / 8 + i)) =
            make_uint4(pack_bf16(x[8 * i] * wgt, x[8 * i + 1] * wgt), pack_bf16(x[8 * i + 2] * wgt, x[8 * i + 3] * wgt),
                       pack_bf16(x[8 * i + 4] * wgt, x[8 * i + 5] * wgt), pack_bf16(x[8 * i + 6] * wgt, x[8 * i + 7] * wgt));
      if (col == 32) {
        fence_async_smem();
        __syncwarp();
        if (lane == 0) tma_store_3d(&tmOut, out_rows, 0, row, bh * args.n_chunks + c);
      }
    };
    // fp32 sum of the segment up to and including chunk c: 32 columns are as many bytes
    auto put_local = [&](int c, int col, const float (&x)[32]) {
      if (lane == 0) bulk_wait_read();
      __syncwarp();
#pragma unroll
      for (int i = 0; i < 8; ++i)
        *reinterpret_cast<float4*>(out_rows + sw128_offset(lane, i)) = make_float4(x[4 * i], x[4 * i + 1], x[4 * i + 2], x[4 * i + 3]);
      fence_async_smem();
      __syncwarp();
      if (lane == 0) tma_store_3d(&tmOut, out_rows, col, row, bh * args.n_chunks + c);
    };
    auto put_z = [&](int c, float z) { args.z[((size_t)bh * args.n_chunks + c) * ROWS + row] = __float2bfloat16_rn(z * wgt); };
    auto put_f32 = [&](float* dst, const float (&x)[32], float f) {
#pragma unroll
      for (int i = 0; i < 8; i += 2) {
        const float4 lo = make_float4(x[4 * i] * f, x[4 * i + 1] * f, x[4 * i + 2] * f, x[4 * i + 3] * f);
        const float4 hi = make_float4(x[4 * i + 4] * f, x[4 * i + 5] * f, x[4 * i + 6] * f, x[4 * i + 7] * f);
        if (args.wide_final) {
          st_global_v8(dst + 4 * i, lo, hi);
        } else {
          reinterpret_cast<float4*>(dst)[i] = lo;
          reinterpret_cast<float4*>(dst)[i + 1] = hi;
        }
      }
    };
    if (first) {
      // the state handed in: into the accumulators, and out in bf16 for chunk 0
      const float inv = (args.packed && a != b) ? 0.70710678118654752440f : 1.f;   // packed rows off the diagonal carry sqrt(2)
      const float4* src = reinterpret_cast<const float4*>(args.s_init + ((size_t)bh * n_pub + prow) * D);
#pragma unroll
      for (int col = 0; col < 64; col += 32) {
        float x[32];
        uint32_t u[32];
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          const float4 y = src[col / 4 + i];
          x[4 * i] = y.x * inv; x[4 * i + 1] = y.y * inv; x[4 * i + 2] = y.z * inv; x[4 * i + 3] = y.w * inv;
        }
#pragma unroll
        for (int i = 0; i < 32; ++i) u[i] = __float_as_uint(x[i]);
        tmem_st32(ta + col, u);
        uint4* dst = reinterpret_cast<uint4*>(args.s + ((size_t)bh * args.n_chunks * ROWS + row) * D + col);
#pragma unroll
        for (int i = 0; i < 4; ++i)
          dst[i] = make_uint4(pack_bf16(x[8 * i] * wgt, x[8 * i + 1] * wgt), pack_bf16(x[8 * i + 2] * wgt, x[8 * i + 3] * wgt),
                              pack_bf16(x[8 * i + 4] * wgt, x[8 * i + 5] * wgt), pack_bf16(x[8 * i + 6] * wgt, x[8 * i + 7] * wgt));
      }
      const float z = args.z_init[(size_t)bh * n_pub + prow] * inv;
      uint32_t u[16] = {__float_as_uint(z)};
      tmem_st16(ta + 64, u);
      put_z(0, z);
      tmem_wait_st();
      tc_fence_before();
      mbar_arrive(bar(BAR_CFREE));
    }
    // (advanced in place: no thread writes before all have read; a row is read and written by one CTA)
    if (args.s_init != nullptr && args.s_final != nullptr) asm volatile("bar.sync 1, 256;" ::: "memory");
    for (int c = c_beg, i = 0; c < c_end && ok; ++c, ++i) {
      ok = wait_or_abort(bar(BAR_CFULL), i & 1, abort_flag);
      if (!ok) break;
      tc_fence_after();
      const bool last = c + 1 == args.n_chunks, fin = last && args.s_final != nullptr;
      uint32_t u[32], zz[4];
#pragma unroll
      for (int col = 0; col < 64; col += 32) {
        tmem_ld32(ta + col, u);
        if (col == 0) tmem_ld4(ta + 64, zz);
        tmem_wait_ld(u);
        if (col == 0) tmem_wait_ld(zz);
        if (col == 32) {
          tc_fence_before();
          mbar_arrive(bar(BAR_CFREE));
        }
        float x[32];
#pragma unroll
        for (int y = 0; y < 32; ++y) x[y] = __uint_as_float(u[y]);
        if (args.s_loc != nullptr) put_local(c, col, x);
        else if (!last) put_state(c + 1, col, x);
        if (fin) {
          // both triangles of a direct state; inside a diagonal block both (a, b) and (b, a) have a thread of their own
          float* dst = args.s_final + (size_t)bh * n_pub * D + col;
          if (args.packed) {
            if (mirror || a <= b) put_f32(dst + (size_t)prow * D, x, a != b ? 1.41421356237309504880f : 1.f);
          } else {
            put_f32(dst + (size_t)public_row<G>(a, b, 0) * D, x, 1.f);
            if (mirror) put_f32(dst + (size_t)public_row<G>(b, a, 0) * D, x, 1.f);
          }
        }
      }
      const float z = __uint_as_float(zz[0]);
      if (args.s_loc != nullptr) args.z_loc[((size_t)bh * args.n_chunks + c) * ROWS + row] = z;
      else if (!last) put_z(c + 1, z);
      if (fin) {
        if (args.packed) {
          if (mirror || a <= b) args.z_final[(size_t)bh * n_pub + prow] = a != b ? z * 1.41421356237309504880f : z;
        } else {
          args.z_final[(size_t)bh * n_pub + public_row<G>(a, b, 0)] = z;
          if (mirror) args.z_final[(size_t)bh * n_pub + public_row<G>(b, a, 0)] = z;
        }
      }
    }
  }

  if (warp >= WARP_CPY0 && lane == 0) bulk_wait();
  // ---------------- teardown ----------------
  if (!ok && args.device_status != nullptr) atomicExch(args.device_status, (int)KATA_ERR_DEVICE_TIMEOUT);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  if (warp == 1 && elect_one()) {
    mma_commit(bar(BAR_DRAIN));
    mbar_wait(bar(BAR_DRAIN), 0);
  }
  __syncthreads();
  if (warp == 0) tmem_dealloc(tb, TMEM_COLS);
}

// Several segments: state before chunk c + 1 = sum of the whole segments before c's + the running sum of c's segment
// (the first one's starts from the state handed in); after the last chunk, the state handed out.
// One thread per (head, state row, four value columns) walks the chunks; eight loads in flight.  Memory-bound: 256 bytes
// read and 128 written per chunk and state row.
template <int G, int R>
__global__ void __launch_bounds__(256) state_fix_kernel(const float* __restrict__ s_loc, const float* __restrict__ z_loc,
                                                        __nv_bfloat16* __restrict__ s, __nv_bfloat16* __restrict__ z, int n_chunks,
                                                        int seg_chunks, float* __restrict__ s_final, float* __restrict__ z_final, int packed) {
  constexpr int ROWS = PairTable<G, R>::kRows;
  static constexpr PairTable<G, R> kPairs{};
  cudaTriggerProgrammaticLaunchCompletion();
  cudaGridDependencySynchronize();
  const int bh = blockIdx.y, idx = blockIdx.x * 256 + threadIdx.x, row = idx >> 4, c4 = idx & 15;   // ROWS is a multiple of 16
  const int p = row >> 6, e = row & 63;
  const int a = 8 * kPairs.g[p] + (e & 7), b = 8 * kPairs.h[p] + (e >> 3);
  const bool mirror = kPairs.g[p] != kPairs.h[p];
  const float wgt = mirror ? 2.f : 1.f;
  float4 off = make_float4(0.f, 0.f, 0.f, 0.f);
  float zoff = 0.f;
  const size_t slot0 = (size_t)bh * n_chunks;
  const int n_sums = s_final != nullptr ? n_chunks : n_chunks - 1;
  constexpr int UNR = 8;
  for (int c0 = 0; c0 < n_sums; c0 += UNR) {
    float4 x[UNR];
    float zx[UNR];
#pragma unroll
    for (int u = 0; u < UNR; ++u)
      if (c0 + u < n_sums) {
        x[u] = reinterpret_cast<const float4*>(s_loc)[((slot0 + c0 + u) * ROWS + row) * 16 + c4];
        zx[u] = c4 == 0 ? z_loc[(slot0 + c0 + u) * ROWS + row] : 0.f;
      }
#pragma unroll
    for (int u = 0; u < UNR; ++u) {
      const int c = c0 + u;
      if (c >= n_sums) break;
      const float4 y = make_float4(off.x + x[u].x, off.y + x[u].y, off.z + x[u].z, off.w + x[u].w);
      const float zy = zoff + zx[u];
      if (c + 1 < n_chunks) {
        reinterpret_cast<uint2*>(s)[((slot0 + c + 1) * ROWS + row) * 16 + c4] =
            make_uint2(pack_bf16(y.x * wgt, y.y * wgt), pack_bf16(y.z * wgt, y.w * wgt));
        if (c4 == 0) z[(slot0 + c + 1) * ROWS + row] = __float2bfloat16_rn(zy * wgt);
      } else {
        const size_t n_pub = public_rows<G>(packed);
        auto put = [&](int r, float f) {
          reinterpret_cast<float4*>(s_final)[((size_t)bh * n_pub + r) * 16 + c4] = make_float4(y.x * f, y.y * f, y.z * f, y.w * f);
          if (c4 == 0) z_final[(size_t)bh * n_pub + r] = zy * f;
        };
        if (packed) {
          if (mirror || a <= b) put(public_row<G>(min(a, b), max(a, b), 1), a != b ? 1.41421356237309504880f : 1.f);
        } else {
          put(public_row<G>(a, b, 0), 1.f);
          if (mirror) put(public_row<G>(b, a, 0), 1.f);
        }
      }
      if ((c + 1) % seg_chunks == 0) {
        off = y;
        zoff = zy;
      }
    }
  }
}

}  // namespace

int tc_state_rows(const Problem& p) {
  return p.groups == 2 ? PairTable<2>::kRows : p.groups == 4 ? PairTable<4>::kRows : tc_narrow(p) ? PairTable<1, 4>::kRows : PairTable<1>::kRows;
}

void tc_states(const Problem& p, const float* rscale, const StatePlan& plan, const StateBuffers& buf, int* device_status,
               LaunchCtx& ctx) {
  const int BH = p.B * p.H;
  const bool segmented = plan.segments > 1;
  CUtensorMap tmK, tmV, tmOut;                    // (tmOut: what goes out per chunk, 128 bytes of 32 rows at a time)
  if (!make_tile_map(&tmK, p.k, BH, p.T, CT, p.d_k) || !make_tile_map(&tmV, p.v, BH, p.T, CT, p.d_v) ||
      !(segmented ? make_tile_map_f32(&tmOut, buf.s_loc, BH * plan.n_chunks, tc_state_rows(p), 32)
                  : make_tile_map(&tmOut, buf.s, BH * plan.n_chunks, tc_state_rows(p), 32))) {
    ctx.status = KATA_ERR_CUDA;
    return;
  }
  const bool narrow = tc_narrow(p);
  auto kern = p.groups == 2 ? tc_state_kernel<2, 8> : p.groups == 4 ? tc_state_kernel<4, 8> : narrow ? tc_state_kernel<1, 4> : tc_state_kernel<1, 8>;
  if (!(p.groups == 2   ? allow_smem<tc_state_kernel<2, 8>>((int)SMEM_ALLOC)
        : p.groups == 4 ? allow_smem<tc_state_kernel<4, 8>>((int)SMEM_ALLOC)
        : narrow        ? allow_smem<tc_state_kernel<1, 4>>((int)SMEM_ALLOC)
                        : allow_smem<tc_state_kernel<1, 8>>((int)SMEM_ALLOC))) {
    ctx.status = KATA_ERR_CUDA;
    return;
  }
  SArgs a{};
  a.rscale = rscale;
  a.s = buf.s;
  a.z = buf.z;
  a.s_loc = segmented ? buf.s_loc : nullptr;
  a.z_loc = segmented ? buf.z_loc : nullptr;
  a.s_init = buf.s_init;
  a.z_init = buf.z_init;
  a.s_final = segmented ? nullptr : buf.s_final;
  a.z_final = segmented ? nullptr : buf.z_final;
  a.wide_final = (reinterpret_cast<uintptr_t>(a.s_final) & 31) == 0;
  a.packed = buf.layout == KATA_LAYOUT_PACKED;
  a.device_status = device_status;
  a.Tlen = p.T;
  a.chunk_tiles = plan.chunk_tokens / CT;
  a.n_chunks = plan.n_chunks;
  a.walk_chunks = buf.s_final != nullptr ? plan.n_chunks : plan.n_chunks - 1;
  a.seg_chunks = plan.seg_chunks;
  const int slices = tc_state_rows(p) / 256;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(slices, BH, plan.segments);
  cfg.blockDim = dim3(NTHREADS);
  cfg.dynamicSmemBytes = SMEM_ALLOC;
  cfg.stream = ctx.stream;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  if (cudaLaunchKernelEx(&cfg, kern, tmK, tmV, tmOut, a) != cudaSuccess) {
    cudaGetLastError();
    ctx.status = KATA_ERR_CUDA;
    return;
  }
  ++ctx.launches;
  if (!segmented) return;
  auto fix = p.groups == 2 ? state_fix_kernel<2, 8> : p.groups == 4 ? state_fix_kernel<4, 8> : narrow ? state_fix_kernel<1, 4> : state_fix_kernel<1, 8>;
  cfg.gridDim = dim3(tc_state_rows(p) / 16, BH);
  cfg.blockDim = dim3(256);
  cfg.dynamicSmemBytes = 0;
  if (cudaLaunchKernelEx(&cfg, fix, (const float*)buf.s_loc, (const float*)buf.z_loc, buf.s, buf.z, plan.n_chunks, plan.seg_chunks,
                         buf.s_final, buf.z_final, (int)(buf.layout == KATA_LAYOUT_PACKED)) != cudaSuccess) {
    cudaGetLastError();
    ctx.status = KATA_ERR_CUDA;
    return;
  }
  ++ctx.launches;
}

}  // namespace kata
