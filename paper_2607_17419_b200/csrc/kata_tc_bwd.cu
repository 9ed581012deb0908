// Backward of the quadratic form on the Blackwell tensor cores: bf16, d_k = d_v = 64, full or blockwise rank-one feature.
//
// With s_ti = q_t . k_i, r_i = 1/||k_i||^2, a_ti = r_i s_ti^2 (i <= t), D_t = sum_i a_ti, o_t = sum_i a_ti v_i / D_t:
//   c_ti = dout_t . v_i,   g_ti = (c_ti - dout_t . o_t) / D_t,   p_ti = s_ti^2 / D_t
//   dq_t = sum_i 2 g_ti s_ti r_i k_i
//   dv_i = r_i sum_t p_ti dout_t
//   dk_i = r_i (u_i - r_i (k_i . u_i) k_i),  u_i = sum_t 2 g_ti s_ti q_t     (the second term is the derivative of r_i; it
//                                                                       makes dk_i orthogonal to k_i: o has degree 0 in k_i)
// A pre-pass writes r; then one kernel in two modes, both with a fixed tile of 128 rows on the TMEM lanes and tiles of NT
// rows streamed past it:
//   MODE_DQ   fixed = 128 queries (Q, dout), streamed = keys (K, V, r), twice:  S = Q K^T, C = dout V^T (SS MMAs); in the
//             first sweep the weight warps sum D_t = sum_i r_i s^2 and sum_i r_i s^2 c in fp32 (the same weights in both,
//             so dout_t . o_t is consistent with c: their difference is what the gradient is made of) and leave
//             (1/D_t, dout_t . o_t) in the workspace; in the second sweep they form E = (c - dout.o) r s, and dq += E K
//             (A = E from TMEM; the row factor 2/D_t in the epilogue)
//   MODE_DKV  fixed = 128 keys (K, V), streamed = queries (Q, dout, their scalars):  S^T = K Q^T, C^T = V dout^T,
//             the weight warps form P^T and E^T with the scalars of the columns, then dv~ += P^T dout, u += E^T Q
//             (B = the streamed tiles read MN-major), and the epilogue applies r_i and the projection.
// No atomics, every sum in a fixed order.
//
// NS = bf16 terms of the weights P and E.  One: kata_bwd_quadratic.  Three (24 bits: fp32 weights; every other operand is
// a bf16 input, exact, and every sum fp32): kata_bwd_chunked on sequences short enough for the quadratic form, whose
// contract is fp32 arithmetic.  Its rows of q and k come as copies scaled by powers of two (exact) to largest entries of 1 to 2,
// so that rows of any norm whose square fp32 holds give the gradients that the walk over the chunks, which normalises
// them, gives; the gradients are scaled back where they are stored.
//
// What bounds it.  A step (128 x 64 pairs) is 256 to 384 cycles of score MMAs and 128 (dq) or 256 (dk, dv) of output MMAs;
// the rest is hand-offs, about 300 cycles each from one thread's arrival through the MMAs to the next thread's first
// instruction.  Where TMEM has room (one group; three terms: dq only) the weights have columns of their own: a score buffer
// is free as soon as its weight warps have read it, so scores, weights and outputs of successive steps overlap; with the
// weights stored over the scores the loop scores -> weights -> outputs -> scores was 2100 cycles for two steps.  Scores and
// outputs are issued by a thread each (an issuer is busy about as long as its MMAs take).  The fixed tiles of dq are TMEM
// operands: from shared memory every score MMA read 6 KB for 32 cycles of arithmetic.  The CTAs are persistent (one per SM,
// items dealt heaviest first, forwards and backwards in turn); the score issuer runs ahead into the next item.
//
// Warps: 0 TMA producer, 1 score MMAs, 2 output MMAs, 3 scalars of the streamed rows, 4.. weights and epilogue (sets of
// four, quadrant = warp % 4; CS sets per buffer, each with its part of the columns).  All waits are bounded.
#include <cuda.h>
#include <type_traits>

#include "kata_common.cuh"
#include "kata_tmap.cuh"
#include "kata_umma.cuh"

namespace kata {
namespace {

using namespace umma;

constexpr int D = 64;
constexpr int MT = 128;          // rows of the fixed tile (TMEM lanes)
constexpr int NSTAGE = 6;
constexpr int WARP_BLD0 = 4;
enum { MODE_DQ = 0, MODE_DKV = 1 };

constexpr uint32_t TMEM_COLS = 512;

// G feature groups of the blockwise map: s_g = q_g . k_g per group, a = r sum_g s_g^2, e_g from s_g; dq and u are formed
// group by group (N = 64 / G columns of the accumulator, the B operand offset into the 128-byte rows).
template <int MODE, int G, int NS> struct Geo {
  static constexpr int NT = G == 4 ? 32 : 64;               // rows of a streamed tile
  static constexpr int NBUF = 2;                            // score buffers
  static constexpr int CS = G == 1 ? 2 : 1;                 // sets of weight warps per buffer
  static constexpr int SETS = NBUF * CS;
  static constexpr int CPW = NT / 32 / CS;                  // runs of 32 columns per set
  static constexpr bool SEP = G == 1 && !(NS == 3 && MODE == MODE_DKV);   // weights in columns of their own
  // a score buffer: [S_0 | .. | S_{G-1} | C], NT fp32 columns each (and 64 more for the extra terms of the weights)
  static constexpr uint32_t BW = SEP ? 128u : NS == 3 ? 192u : (uint32_t)(G + 1) * NT;
  static constexpr uint32_t CB = G * NT;                    // its C block
  static constexpr uint32_t EW = MODE == MODE_DQ ? 32 * NS : 64;          // SEP: columns of the weights of a buffer, from 256 on
  static constexpr bool XT = SEP && MODE == MODE_DQ && NS == 1;           // fixed tiles in TMEM, two buffers of 64 columns
  static constexpr uint32_t COL_X = 384;
  static constexpr uint32_t COL_ACC = SEP ? 256 + NBUF * EW : 384;        // accumulators: 64 or 128 columns
  static constexpr int NTHREADS = 128 + SETS * 128;
  static_assert(NBUF * BW <= (SEP ? 256u : COL_ACC) && COL_ACC + (MODE == MODE_DQ ? 64 : 128) <= (XT ? COL_X : 512u), "TMEM columns");
  // first of the 16 columns of the bf16 weights of 32 streamed rows (run ch of a buffer): columns of their own, or over scores
  // that the same warp has in its registers (three terms: P and E of a term side by side, over the run's columns of S, of C
  // and of the 64 more, so that no set touches what the other still reads)
  __host__ __device__ static constexpr uint32_t p_col(int b, int term, int ch) {
    return SEP ? 256 + b * EW + ch * 16 : b * BW + (NS == 3 ? term * 64 + ch * 32 : CB + ch * 16);
  }
  __host__ __device__ static constexpr uint32_t e_col(int b, int g, int term, int ch) {
    return SEP ? 256 + b * EW + (MODE == MODE_DQ ? 32 * term : 32) + ch * 16 : b * BW + (NS == 3 ? term * 64 + ch * 32 + 16 : g * NT + ch * 16);
  }
};

// Registers with 640 threads: 96 each at launch; the four warps that issue and copy give theirs to the weight warps.
template <int N> __device__ __forceinline__ void regs_release() { asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(N)); }
template <int N> __device__ __forceinline__ void regs_take() { asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(N)); }
static_assert(128 * 64 + 512 * 104 <= 640 * 96, "register budget");

constexpr uint32_t OFF_X = 0;                      // 2 x (two fixed tiles of 128 x 64 bf16, 128B swizzle): this and the next item
constexpr uint32_t OFF_ST = 65536;                 // stages: two streamed tiles of up to 8 KB
constexpr uint32_t STAGE_BYTES = 16384;
constexpr uint32_t OFF_SC = OFF_ST + NSTAGE * STAGE_BYTES;   // per stage 512 bytes of scalars of the streamed rows:
                                                             // r_i (MODE_DQ) or 1/D_t and -dout_t . o_t (MODE_DKV)
constexpr uint32_t OFF_PART = OFF_SC + NSTAGE * 512;         // 2 (item parity) x 4 sets x 128 float2: the sums of a row meet here
constexpr uint32_t OFF_BAR = OFF_PART + 8192;
constexpr uint32_t SMEM_BYTES = OFF_BAR + 256;
constexpr uint32_t SMEM_ALLOC = SMEM_BYTES + 1024;
static_assert(SMEM_ALLOC > 116 * 1024, "one CTA per SM is assumed (the CTA allocates all of TMEM)");

// Every barrier has waiters that consume each of its phases in order; a producer of a phase always depends on the
// waiter's progress (no barrier can complete two phases ahead of a waiter).
enum {
  BAR_XFULL = 0,     // [2] fixed tiles of an item landed
  BAR_XEMPTY = 2,    // [2] ... and are no longer needed
  BAR_FULL = 4,      // [NSTAGE] streamed tiles (TMA bytes) and their scalars landed
  BAR_EMPTY = 10,    // [NSTAGE] stage free
  BAR_SFULL = 16,    // [2] scores in TMEM
  BAR_SFREE = 18,    // [2] the score buffer may take new scores (its weight warps; where weights lie over scores, the output MMAs)
  BAR_PFULL = 20,    // [2] weights stored, scalars read (CS x 128 threads)
  BAR_PFREE = 22,    // [2] weights consumed, or (first sweep) the step seen by the output issuer
  BAR_ODONE = 24,    // the accumulators of an item are complete
  BAR_OFREE = 25,    // ... and have been read (256 threads)
  BAR_XT = 26,       // [2] fixed tiles of an item in TMEM (256 threads)
  BAR_DRAIN = 28,
  BAR_MEET = 29,     // MODE_DQ: the sums of an item are in shared memory (all weight threads)
  BAR_COUNT = 30
};

struct BArgs {
  __nv_bfloat16* out0;       // MODE_DQ: dq;  MODE_DKV: dk
  __nv_bfloat16* out1;       // MODE_DKV: dv
  float* stats;              // [BH][T][2]: 1 / D_t, dout_t . o_t (written by MODE_DQ, read by MODE_DKV)
  const float* rk;           // [BH][T]: 1 / ||k_i||^2
  const float* row_scale;    // NS = 3: [BH][T] power of two that the row of q (MODE_DQ) or k (MODE_DKV) was scaled by
  int* device_status;
  int wide_out;              // rows of the gradients are 32-byte aligned
  int Tlen;
  int BH;
};

__device__ __forceinline__ float2 unpack_bf16(uint32_t x) {
  return make_float2(__uint_as_float(x << 16), __uint_as_float(x & 0xFFFF0000u));
}
// v as the sum of NS pairs of bf16 (three: all 24 bits)
template <int NS> __device__ __forceinline__ void split_pack(float2 v, uint32_t (&t)[NS]) {
#pragma unroll
  for (int i = 0; i < NS; ++i) {
    t[i] = pack_bf16(v.x, v.y);
    if (i + 1 < NS) {
      const float2 u = unpack_bf16(t[i]);
      v = __fadd2_rn(v, make_float2(-u.x, -u.y));
    }
  }
}

__device__ __forceinline__ void st_cols(uint32_t t, const uint32_t (&r)[8]) { tmem_st8(t, r); }
__device__ __forceinline__ void st_cols(uint32_t t, const uint32_t (&r)[16]) { tmem_st16(t, r); }

template <int MODE, int G, int NS>
__global__ void __launch_bounds__(Geo<MODE, G, NS>::NTHREADS, 1)
tc_bwd_kernel(const __grid_constant__ CUtensorMap tmX1, const __grid_constant__ CUtensorMap tmX2,
              const __grid_constant__ CUtensorMap tmY1, const __grid_constant__ CUtensorMap tmY2, const BArgs args) {
  using geo = Geo<MODE, G, NS>;
  constexpr int NT = geo::NT, NBUF = geo::NBUF, CS = geo::CS, CPW = geo::CPW, SETS = geo::SETS;
  constexpr uint32_t BW = geo::BW, CB = geo::CB, COL_ACC = geo::COL_ACC, COL_X = geo::COL_X;
  constexpr bool XT = geo::XT, SEP = geo::SEP;
  constexpr int MG = D / G;                        // features per group
  extern __shared__ unsigned char smem_raw[];
  unsigned char* base = reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  auto bar = [&](int i) { return reinterpret_cast<uint64_t*>(base + OFF_BAR) + i; };
  auto x1 = [&](int b) { return base + OFF_X + b * 32768; };
  auto x2 = [&](int b) { return base + OFF_X + b * 32768 + 16384; };
  auto y1 = [&](int s) { return base + OFF_ST + s * STAGE_BYTES; };
  auto y2 = [&](int s) { return base + OFF_ST + s * STAGE_BYTES + 8192; };
  auto sc = [&](int s) { return base + OFF_SC + s * 512; };
  __shared__ uint32_t tmem_base_s;
  __shared__ int abort_s;
  volatile int* abort_flag = &abort_s;

  cudaTriggerProgrammaticLaunchCompletion();                      // (dk, dv start on the SMs that dq leaves)
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int n_m = (args.Tlen + MT - 1) / MT;                      // fixed tiles of a head
  const int n_stream = (args.Tlen + NT - 1) / NT;                 // streamed tiles of the whole sequence
  const long long n_items = (long long)args.BH * n_m;
  struct Item {
    int bh, m0;
    int jbeg, ntiles;             // streamed tiles
    int nsteps;                   // MODE_DQ streams the keys twice
  };
  // MODE_DQ: heaviest (last) query tiles first, keys 0 .. m0 + 127;  MODE_DKV: the first key tiles are the heaviest,
  // queries m0 .. T - 1.  Rounds of gridDim.x items, dealt forwards and backwards in turn.
  auto next_item = [&](int& n, Item& it) -> bool {   // the item at or after the n-th; n is left at it
    for (;; ++n) {
      if ((long long)n * gridDim.x >= n_items) return false;
      const long long id = (long long)n * gridDim.x + ((n & 1) ? (int)gridDim.x - 1 - (int)blockIdx.x : (int)blockIdx.x);
      if (id >= n_items) continue;
      const int rank = (int)(id / args.BH), mtile = MODE == MODE_DQ ? n_m - 1 - rank : rank;
      it.bh = (int)(id % args.BH);
      it.m0 = mtile * MT;
      it.jbeg = MODE == MODE_DQ ? 0 : mtile * (MT / NT);
      const int jend = MODE == MODE_DQ ? min(n_stream, (mtile + 1) * (MT / NT)) : n_stream;
      it.ntiles = jend - it.jbeg;
      it.nsteps = MODE == MODE_DQ ? 2 * it.ntiles : it.ntiles;
      return true;
    }
  };

  if (tid == 0) {
    abort_s = 0;
    for (int i = 0; i < 2; ++i) {
      mbar_init(bar(BAR_XFULL + i), 1);
      mbar_init(bar(BAR_XEMPTY + i), (MODE == MODE_DQ && !XT ? 0 : 256) + (XT ? 0 : 1));   // readers: sets 0 and 1, MMAs
      mbar_init(bar(BAR_XT + i), 256);
    }
    for (int i = 0; i < NSTAGE; ++i) {
      mbar_init(bar(BAR_FULL + i), 2);
      mbar_init(bar(BAR_EMPTY + i), 1);
    }
    for (int i = 0; i < NBUF; ++i) {
      mbar_init(bar(BAR_SFULL + i), 1);
      mbar_init(bar(BAR_SFREE + i), SEP ? CS * 128 : 1);
      mbar_init(bar(BAR_PFULL + i), CS * 128);
      mbar_init(bar(BAR_PFREE + i), 1);
    }
    mbar_init(bar(BAR_ODONE), 1);
    mbar_init(bar(BAR_OFREE), 256);
    mbar_init(bar(BAR_DRAIN), 2);
    mbar_init(bar(BAR_MEET), SETS * 128);
    fence_mbar_init();
    tma_prefetch_desc(&tmX1);
    tma_prefetch_desc(&tmX2);
    tma_prefetch_desc(&tmY1);
    tma_prefetch_desc(&tmY2);
  }
  if (warp == 0) {
    tmem_alloc(&tmem_base_s, TMEM_COLS);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tb = tmem_base_s;
  bool ok = true;
  // A programmatic dependent launch.  dk, dv start while dq runs on other SMs and wait for it here, where no limit on time
  // applies; dq waits for its pre-pass where it reads the key scales, or, where that writes the rows it loads, here.
  if (MODE == MODE_DKV || NS == 3) cudaGridDependencySynchronize();

  if (warp == 0) {
    if (SETS == 4) regs_release<64>();
    // =========================== TMA producer ===========================
    if (elect_one()) {
      // the fixed tiles of an item are asked for behind the third step of the item before
      uint32_t t = 0;
      int ni = 0;
      Item w, wn;
      int n = 0;
      auto load_x = [&](const Item& x, int i) {
        const int xb = i & 1;
        ok = wait_or_abort(bar(BAR_XEMPTY + xb), ((i >> 1) & 1) ^ 1, abort_flag);
        if (!ok) return;
        mbar_arrive_expect_tx(bar(BAR_XFULL + xb), 32768);
        tma_load_3d(x1(xb), &tmX1, bar(BAR_XFULL + xb), 0, x.m0, x.bh);
        tma_load_3d(x2(xb), &tmX2, bar(BAR_XFULL + xb), 0, x.m0, x.bh);
      };
      bool more = next_item(n, w);
      if (more) load_x(w, 0);
      for (; more && ok; ++ni) {
        ++n;
        const bool more_n = next_item(n, wn);
        for (int j = 0, jt = 0; j < w.nsteps && ok; ++j, ++t) {
          const int s = t % NSTAGE;
          ok = wait_or_abort(bar(BAR_EMPTY + s), ((t / NSTAGE) & 1) ^ 1, abort_flag);
          if (!ok) break;
          mbar_arrive_expect_tx(bar(BAR_FULL + s), 2 * NT * 128);
          tma_load_3d(y1(s), &tmY1, bar(BAR_FULL + s), 0, (w.jbeg + jt) * NT, w.bh);
          tma_load_3d(y2(s), &tmY2, bar(BAR_FULL + s), 0, (w.jbeg + jt) * NT, w.bh);
          if (++jt == w.ntiles) jt = 0;
          if (more_n && j == (w.nsteps > 2 ? 2 : w.nsteps - 1)) load_x(wn, ni + 1);
        }
        w = wn;
        more = more_n;
      }
    }
  } else if (warp == 1) {
    if (SETS == 4) regs_release<64>();
    // =========================== score MMA issuer ===========================
    if (elect_one()) {
      const uint32_t id_s = instr_desc(kFmtBF16, kFmtBF16, 0, 0, 128, NT);      // both K-major
      const uint64_t dk = smem_desc(0, 16, 1024, kSwizzle128B), dy = at(dk, smem_u32(y1(0)));
      uint32_t t = 0;
      int ni = 0;
      Item w;
      for (int n = 0; ok && next_item(n, w); ++n, ++ni) {
        const int xb = ni & 1;
        ok = wait_or_abort(bar((XT ? BAR_XT : BAR_XFULL) + xb), (ni >> 1) & 1, abort_flag);
        const uint64_t f1 = at(dk, smem_u32(x1(xb)));
        const uint32_t xt = tb + COL_X + xb * 64;
        for (int j = 0; j < w.nsteps && ok; ++j, ++t) {
          const int s = t % NSTAGE, b = t % NBUF;
          ok = wait_or_abort(bar(BAR_FULL + s), (t / NSTAGE) & 1, abort_flag) &&
               wait_or_abort(bar(BAR_SFREE + b), ((t / NBUF) & 1) ^ 1, abort_flag);
          if (!ok) break;
          tc_fence_after();
          const uint64_t a1 = dy + s * (STAGE_BYTES / 16), a2 = a1 + 8192 / 16, f2 = f1 + 16384 / 16;
#pragma unroll
          for (int ks = 0; ks < 4; ++ks) {    // 16 features per step; group ks / (4 / G) has its own NT score columns
            const uint32_t d = tb + b * BW + (ks / (4 / G)) * NT;
            if (XT) mma_f16_ts(d, xt + ks * 8, a1 + ks * 2, id_s, (ks % (4 / G)) > 0);
            else mma_f16_ss(d, f1 + ks * 2, a1 + ks * 2, id_s, (ks % (4 / G)) > 0);
          }
#pragma unroll
          for (int ks = 0; ks < 4; ++ks) {
            const uint32_t d = tb + b * BW + CB;
            if (XT) mma_f16_ts(d, xt + 32 + ks * 8, a2 + ks * 2, id_s, ks > 0);
            else mma_f16_ss(d, f2 + ks * 2, a2 + ks * 2, id_s, ks > 0);
          }
          mma_commit(bar(BAR_SFULL + b));
        }
        if (!XT && ok) mma_commit(bar(BAR_XEMPTY + xb));
      }
    }
  } else if (warp == 2) {
    if (SETS == 4) regs_release<64>();
    // =========================== output MMA issuer ===========================
    if (elect_one()) {
      const uint32_t id_o = instr_desc(kFmtBF16, kFmtBF16, 0, 1, 128, 64);      // dv~: A tmem, B MN-major
      const uint32_t id_g = instr_desc(kFmtBF16, kFmtBF16, 0, 1, 128, MG);      // dq, u of a feature group
      // 8 streamed rows x 64 columns per 1 KB atom
      const uint64_t dmn = at(smem_desc(0, 8192, 1024, kSwizzle128B), smem_u32(y1(0)));
      uint32_t t = 0;
      int ni = 0;
      Item w;
      for (int n = 0; ok && next_item(n, w); ++n, ++ni) {
        uint32_t acc = 0;
        for (int j = 0; j < w.nsteps && ok; ++j, ++t) {
          const int s = t % NSTAGE, b = t % NBUF;
          ok = wait_or_abort(bar(BAR_PFULL + b), (t / NBUF) & 1, abort_flag);
          if (!ok) break;
          if (MODE == MODE_DQ && j < w.ntiles) {         // (the first sweep only sums the row scalars)
            mbar_arrive(bar((SEP ? BAR_PFREE : BAR_SFREE) + b));
            mbar_arrive(bar(BAR_EMPTY + s));
            continue;
          }
          // the accumulators are free once the epilogue of the item before has read them
          if (acc == 0 && ni > 0) ok = wait_or_abort(bar(BAR_OFREE), (ni - 1) & 1, abort_flag);
          if (!ok) break;
          tc_fence_after();
          const uint64_t ya = dmn + s * (STAGE_BYTES / 16), yb = ya + 8192 / 16;
          if (MODE == MODE_DKV) {
#pragma unroll
            for (int term = 0; term < NS; ++term)
#pragma unroll
              for (int ks = 0; ks < NT / 16; ++ks)      // dv~ += P^T dout
                mma_f16_ts(tb + COL_ACC, tb + geo::p_col(b, term, ks / 2) + (ks & 1) * 8, yb + ks * 128, id_o, term > 0 || ks > 0 ? 1u : acc);
          }
          constexpr uint32_t col = COL_ACC + (MODE == MODE_DKV ? 64 : 0);
#pragma unroll
          for (int g = 0; g < G; ++g)
#pragma unroll
            for (int term = 0; term < NS; ++term)
#pragma unroll
              for (int ks = 0; ks < NT / 16; ++ks)      // dq += E K, u += E^T Q
                mma_f16_ts(tb + col + g * MG, tb + geo::e_col(b, g, term, ks / 2) + (ks & 1) * 8, ya + (ks * 128 + g * MG / 8), id_g,
                           term > 0 || ks > 0 ? 1u : acc);
          acc = 1;
          mma_commit(bar((SEP ? BAR_PFREE : BAR_SFREE) + b));
          mma_commit(bar(BAR_EMPTY + s));
        }
        if (ok) mma_commit(bar(BAR_ODONE));
      }
    }
  } else if (warp == 3) {
    if (SETS == 4) regs_release<64>();
    // =========================== scalars of the streamed rows, two tiles ahead ===========================
    if (MODE == MODE_DQ) cudaGridDependencySynchronize();
    constexpr int RPL = NT / 32;                       // rows per lane
    constexpr int FPR = MODE == MODE_DQ ? 1 : 2;       // floats per row
    const float* src = MODE == MODE_DQ ? args.rk : args.stats;
    Item wl, w;
    int nl = 0, jl = 0;
    bool ml = next_item(nl, wl);
    auto fetch = [&](float (&v)[RPL * FPR]) {
#pragma unroll
      for (int e = 0; e < RPL; ++e) {
        const int row = (wl.jbeg + (jl >= wl.ntiles ? jl - wl.ntiles : jl)) * NT + lane * RPL + e;
        const bool in = ml && row < args.Tlen;
#pragma unroll
        for (int f = 0; f < FPR; ++f) v[e * FPR + f] = in ? src[((size_t)wl.bh * args.Tlen + row) * FPR + f] : 0.f;
      }
      if (ml && ++jl == wl.nsteps) {
        jl = 0;
        ++nl;
        ml = next_item(nl, wl);
      }
    };
    float v0[RPL * FPR], v1[RPL * FPR], v2[RPL * FPR];
    fetch(v0);
    fetch(v1);
    uint32_t t = 0;
    for (int n = 0; ok && next_item(n, w); ++n)
      for (int j = 0; j < w.nsteps && ok; ++j, ++t) {
        const int s = t % NSTAGE;
        fetch(v2);
        ok = wait_or_abort(bar(BAR_EMPTY + s), ((t / NSTAGE) & 1) ^ 1, abort_flag);
        if (!ok) break;
#pragma unroll
        for (int e = 0; e < RPL * FPR; ++e) {
          // MODE_DKV: (1/D, 1/D, -dout.o, -dout.o) of a pair of rows, the operands of the packed multiplies and adds
          const int i = lane * RPL * FPR + e, row = i >> 1;
          if (MODE == MODE_DQ) reinterpret_cast<float*>(sc(s))[i] = v0[e];
          else reinterpret_cast<float*>(sc(s))[(row >> 1) * 4 + (i & 1) * 2 + (row & 1)] = (i & 1) ? -v0[e] : v0[e];
          v0[e] = v1[e];
          v1[e] = v2[e];
        }
        __syncwarp();
        if (lane == 0) mbar_arrive(bar(BAR_FULL + s));
      }
  } else if (warp >= WARP_BLD0) {
    if (SETS == 4) regs_take<104>();
    // =========================== weights and epilogue (SETS sets of 128 threads) ===========================
    const uint32_t q4 = warp & 3;
    const int set = (warp - WARP_BLD0) >> 2;
    const int grp = set / CS;                    // this set's buffer: the steps t with t % NBUF = grp
    const int ch0 = set % CS;                    // ... and its columns of every block (CPW runs of 32)
    const int rowl = q4 * 32 + lane;             // row of the fixed tile (= TMEM lane)
    const uint32_t lanes = tmem_addr(tb, q4 * 32, 0), buf = lanes + grp * BW, accu = lanes + COL_ACC;
    // fixed tiles of item i from shared memory to TMEM: set 0 the first, set 1 the second
    auto copy_x = [&](int i) {
      const int xb = i & 1;
      ok = ok && wait_or_abort(bar(BAR_XFULL + xb), (i >> 1) & 1, abort_flag);
      if (!ok) return;
      const unsigned char* src = set == 0 ? x1(xb) : x2(xb);
#pragma unroll
      for (int hf = 0; hf < 2; ++hf) {
        uint32_t r[16];
#pragma unroll
        for (int c = 0; c < 4; ++c) {
          const uint4 v = *reinterpret_cast<const uint4*>(src + sw128_offset(rowl, hf * 4 + c));
          r[4 * c] = v.x; r[4 * c + 1] = v.y; r[4 * c + 2] = v.z; r[4 * c + 3] = v.w;
        }
        tmem_st16(tmem_addr(tb, q4 * 32, COL_X + xb * 64 + set * 32 + hf * 16), r);
      }
      tmem_wait_st();
      tc_fence_before();
      mbar_arrive(bar(BAR_XT + xb));
      if (MODE == MODE_DQ) mbar_arrive(bar(BAR_XEMPTY + xb));
    };
    uint32_t t0 = 0, n_out = 0;                  // steps of the items before; steps of this set's buffer
    int ni = 0;
    Item w, wn;
    int n = 0, nn = 0;
    bool more = next_item(n, w);
    if (XT && more && set < 2) copy_x(0);
    for (; more && ok; ++ni) {
      nn = n + 1;
      const bool more_n = next_item(nn, wn);
      const int grow = w.m0 + rowl;
      float inv_row = 0.f, del_row = 0.f;        // MODE_DQ: the scalars of this query (1 / D_t, dout_t . o_t)
      int j = (grp + NBUF - (int)(t0 % NBUF)) % NBUF;
      auto begin = [&](uint32_t t) -> bool {
        if (!wait_or_abort(bar(BAR_SFULL + grp), (t / NBUF) & 1, abort_flag)) return false;
        tc_fence_after();
        return true;
      };
      auto read_done = [&]() {                   // the scores are in registers
        if (!SEP) return;
        tc_fence_before();
        mbar_arrive(bar(BAR_SFREE + grp));
      };
      auto end = [&]() {
        tc_fence_before();
        mbar_arrive(bar(BAR_PFULL + grp));
      };
      if (MODE == MODE_DQ) {
        // ---- first sweep: a = r_i sum_g s_g^2 for the keys n <= this query; D_t += a, sum += a c ----
        float sum_d = 0.f, sum_m = 0.f;
        for (; j < w.ntiles && ok; j += NBUF) {
          ok = begin(t0 + j);
          if (!ok) break;
          const int s = (t0 + j) % NSTAGE;
#pragma unroll 1
          for (int ch = ch0; ch < ch0 + CPW; ++ch) {
          const int n0 = (w.jbeg + j) * NT + ch * 32;
          const float4* cs = reinterpret_cast<const float4*>(sc(s) + ch * 128);       // r of four keys
          float2 d2 = make_float2(0.f, 0.f), m2 = make_float2(0.f, 0.f);
          // two copies of the loop, chosen once per tile: the causal test exists on diagonal tiles only
          auto sums = [&](auto masked) {
            uint32_t sx[32], cx[32];
            tmem_ld32(buf + ch * 32, sx);
            tmem_ld32(buf + CB + ch * 32, cx);
            tmem_wait_ld(sx);
            tmem_wait_ld(cx);
            read_done();
            float2 ss[G > 1 ? 16 : 1];
            if constexpr (G > 1) {
#pragma unroll
              for (int g = 0; g < G; ++g) {
                if (g > 0) {
                  tmem_ld32(buf + g * NT + ch * 32, sx);
                  tmem_wait_ld(sx);
                }
#pragma unroll
                for (int c = 0; c < 32; c += 2) {
                  const float2 s2 = make_float2(__uint_as_float(sx[c]), __uint_as_float(sx[c + 1]));
                  ss[c / 2] = g == 0 ? __fmul2_rn(s2, s2) : __ffma2_rn(s2, s2, ss[c / 2]);
                }
              }
            }
#pragma unroll
            for (int c = 0; c < 32; c += 4) {
              const float4 r4 = cs[c / 4];
#pragma unroll
              for (int e = 0; e < 4; e += 2) {
                const float2 s2 = make_float2(__uint_as_float(sx[c + e]), __uint_as_float(sx[c + e + 1]));
                float2 a2 = __fmul2_rn(G > 1 ? ss[G > 1 ? (c + e) / 2 : 0] : __fmul2_rn(s2, s2), e == 0 ? make_float2(r4.x, r4.y) : make_float2(r4.z, r4.w));
                if constexpr (decltype(masked)::value) {
                  if (n0 + c + e > grow) a2.x = 0.f;
                  if (n0 + c + e + 1 > grow) a2.y = 0.f;
                }
                d2 = __fadd2_rn(d2, a2);
                m2 = __ffma2_rn(a2, make_float2(__uint_as_float(cx[c + e]), __uint_as_float(cx[c + e + 1])), m2);
              }
            }
          };
          if (n0 + 31 > w.m0) sums(std::true_type{}); else sums(std::false_type{});
          sum_d += d2.x + d2.y;
          sum_m += m2.x + m2.y;
          }
          // (nothing is stored, but the output issuer must have seen this buffer's step before: a parity cannot tell two
          // phases of BAR_PFULL apart)
          if (SEP && n_out > 0) ok = wait_or_abort(bar(BAR_PFREE + grp), (n_out - 1) & 1, abort_flag);
          if (!ok) break;
          ++n_out;
          end();
        }
        if (!ok) break;
        // the sets' shares of a row meet, in a fixed order (a bounded wait: a set that has given up does not come)
        float2* part = reinterpret_cast<float2*>(base + OFF_PART) + (ni & 1) * 512 + rowl;
        part[set * MT] = make_float2(sum_d, sum_m);
        mbar_arrive(bar(BAR_MEET));
        ok = wait_or_abort(bar(BAR_MEET), ni & 1, abort_flag);
        if (!ok) break;
        float dt = 0.f, mt = 0.f;
#pragma unroll
        for (int g = 0; g < SETS; ++g) {
          dt += part[g * MT].x;
          mt += part[g * MT].y;
        }
        inv_row = dt > 0.f ? 1.f / dt : 0.f;
        del_row = mt * inv_row;
        if (set == 0 && grow < args.Tlen)
          *reinterpret_cast<float2*>(args.stats + ((size_t)w.bh * args.Tlen + grow) * 2) = make_float2(inv_row, del_row);
      }
      // ---- weights ----
      for (; j < w.nsteps && ok; j += NBUF) {
        ok = begin(t0 + j);
        if (!ok) break;
        const int s = (t0 + j) % NSTAGE;
#pragma unroll
        for (int cc = 0; cc < CPW; ++cc) {
        const int ch = ch0 + cc;
        const int n0 = (w.jbeg + (MODE == MODE_DQ ? j - w.ntiles : j)) * NT + ch * 32;
        auto dead = [&](int c) { return MODE == MODE_DQ ? n0 + c > grow : n0 + c < grow; };
        const bool diag = MODE == MODE_DQ ? n0 + 31 > w.m0 : n0 < w.m0 + MT - 1;
        const float4* cs = reinterpret_cast<const float4*>(sc(s) + ch * (MODE == MODE_DQ ? 128 : 256));
        if constexpr (G == 1) {
          // e = (c - dout.o) r s, or (c - dout_t.o_t) s / D_t with p = s^2 / D_t
          auto weigh = [&](auto masked) {
            constexpr int CW = 16;
            uint32_t sv[32], cv[32];
            tmem_ld32(buf + ch * 32, sv);
            tmem_ld32(buf + CB + ch * 32, cv);
            tmem_wait_ld(sv);
            tmem_wait_ld(cv);
            read_done();
#pragma unroll
            for (int c0 = 0; c0 < 32; c0 += CW) {
              uint32_t pe[NS][CW / 2], pp[MODE == MODE_DKV ? NS : 1][CW / 2];
#pragma unroll
              for (int c = c0; c < c0 + CW; c += 2) {
                const float2 s2 = make_float2(__uint_as_float(sv[c]), __uint_as_float(sv[c + 1]));
                const float2 c2 = make_float2(__uint_as_float(cv[c]), __uint_as_float(cv[c + 1]));
                float2 e2, p2 = make_float2(0.f, 0.f);
                if (MODE == MODE_DQ) {
                  const float4 r4 = cs[c / 4];
                  e2 = __fmul2_rn(__fmul2_rn(__fadd2_rn(c2, make_float2(-del_row, -del_row)), (c & 2) ? make_float2(r4.z, r4.w) : make_float2(r4.x, r4.y)), s2);
                } else {
                  const float4 st = cs[c / 2];                                  // 1/D and -dout.o of two queries
                  const float2 t2 = __fmul2_rn(s2, make_float2(st.x, st.y));    // s / D
                  p2 = __fmul2_rn(t2, s2);
                  e2 = __fmul2_rn(__fadd2_rn(c2, make_float2(st.z, st.w)), t2);
                }
                if constexpr (decltype(masked)::value) {
                  if (dead(c)) { e2.x = 0.f; p2.x = 0.f; }
                  if (dead(c + 1)) { e2.y = 0.f; p2.y = 0.f; }
                }
                uint32_t term[NS];
                split_pack<NS>(e2, term);
#pragma unroll
                for (int i = 0; i < NS; ++i) pe[i][(c - c0) / 2] = term[i];
                if constexpr (MODE == MODE_DKV) {
                  split_pack<NS>(p2, term);
#pragma unroll
                  for (int i = 0; i < NS; ++i) pp[i][(c - c0) / 2] = term[i];
                }
              }
              // the outputs of two steps back have read this buffer's weights; waited for with the first half of the new ones in
              // registers (before them: dq 415 -> 406 us, dk dv 324 -> 300, 64 heads x 4096)
              if (SEP && c0 == 0 && n_out > 0) ok = wait_or_abort(bar(BAR_PFREE + grp), (n_out - 1) & 1, abort_flag);
              if (!ok) return;
#pragma unroll
              for (int i = 0; i < NS; ++i) {
                st_cols(lanes + geo::e_col(grp, 0, i, ch) + c0 / 2, pe[i]);
                if constexpr (MODE == MODE_DKV) st_cols(lanes + geo::p_col(grp, i, ch) + c0 / 2, pp[i]);
              }
            }
          };
          if (diag) weigh(std::true_type{}); else weigh(std::false_type{});
        } else {
          uint32_t sv[32], cv[32];
          tmem_ld32(buf + ch * 32, sv);
          tmem_ld32(buf + CB + ch * 32, cv);
          tmem_wait_ld(sv);
          tmem_wait_ld(cv);
          // f: e = f s, over c in place
          auto factors = [&](auto masked) {
#pragma unroll
            for (int c = 0; c < 32; c += 2) {
              const float2 c2 = make_float2(__uint_as_float(cv[c]), __uint_as_float(cv[c + 1]));
              float2 f;
              if (MODE == MODE_DQ) {
                const float4 r4 = cs[c / 4];
                f = __fmul2_rn(__fadd2_rn(c2, make_float2(-del_row, -del_row)), (c & 2) ? make_float2(r4.z, r4.w) : make_float2(r4.x, r4.y));
              } else {
                const float4 st = cs[c / 2];
                f = __fmul2_rn(__fadd2_rn(c2, make_float2(st.z, st.w)), make_float2(st.x, st.y));
              }
              if constexpr (decltype(masked)::value) {
                if (dead(c)) f.x = 0.f;
                if (dead(c + 1)) f.y = 0.f;
              }
              cv[c] = __float_as_uint(f.x);
              cv[c + 1] = __float_as_uint(f.y);
            }
          };
          if (diag) factors(std::true_type{}); else factors(std::false_type{});
          float2 ss[MODE == MODE_DKV ? 16 : 1];
          uint32_t pk[16];
#pragma unroll
          for (int g = 0; g < G; ++g) {
            if (g > 0) {
              tmem_ld32(buf + g * NT + ch * 32, sv);
              tmem_wait_ld(sv);
            }
#pragma unroll
            for (int c = 0; c < 32; c += 2) {
              const float2 s2 = make_float2(__uint_as_float(sv[c]), __uint_as_float(sv[c + 1]));
              if constexpr (MODE == MODE_DKV) ss[c / 2] = g == 0 ? __fmul2_rn(s2, s2) : __ffma2_rn(s2, s2, ss[c / 2]);
              const float2 e2 = __fmul2_rn(make_float2(__uint_as_float(cv[c]), __uint_as_float(cv[c + 1])), s2);
              pk[c / 2] = pack_bf16(e2.x, e2.y);
            }
            tmem_st16(lanes + geo::e_col(grp, g, 0, ch), pk);
          }
          if constexpr (MODE == MODE_DKV) {
            // p = sum_g s_g^2 / D_t
            auto weights = [&](auto masked) {
#pragma unroll
              for (int c = 0; c < 32; c += 2) {
                const float4 st = cs[c / 2];
                float2 p2 = __fmul2_rn(ss[c / 2], make_float2(st.x, st.y));
                if constexpr (decltype(masked)::value) {
                  if (dead(c)) p2.x = 0.f;
                  if (dead(c + 1)) p2.y = 0.f;
                }
                pk[c / 2] = pack_bf16(p2.x, p2.y);
              }
            };
            if (diag) weights(std::true_type{}); else weights(std::false_type{});
            tmem_st16(lanes + geo::p_col(grp, 0, ch), pk);
          }
        }
        }
        if (!ok) break;
        tmem_wait_st();
        ++n_out;
        end();
      }
      t0 += w.nsteps;
      // the next item's fixed tiles go to TMEM (the item before, in the same buffer, is complete) before the wait for this
      // item's last MMAs
      if (XT && set < 2 && more_n && ok) copy_x(ni + 1);
      const Item cur = w;
      n = nn;
      w = wn;
      more = more_n;
      if (!ok) break;
      if (set > 1) continue;
      // ---- epilogue: sets 0 and 1 ----
      ok = wait_or_abort(bar(BAR_ODONE), ni & 1, abort_flag) &&
           (MODE == MODE_DQ || wait_or_abort(bar(BAR_XFULL + (ni & 1)), (ni >> 1) & 1, abort_flag));   // (k is read below)
      if (!ok) break;
      tc_fence_after();
      auto store32 = [&](__nv_bfloat16* dst, const float (&x)[32]) {
#pragma unroll
        for (int c = 0; c < 32; c += 16) {
          uint4 pkt[2];
#pragma unroll
          for (int e = 0; e < 2; ++e)
            pkt[e] = make_uint4(pack_bf16(x[c + 8 * e], x[c + 8 * e + 1]), pack_bf16(x[c + 8 * e + 2], x[c + 8 * e + 3]),
                                pack_bf16(x[c + 8 * e + 4], x[c + 8 * e + 5]), pack_bf16(x[c + 8 * e + 6], x[c + 8 * e + 7]));
          store_32(dst + c, pkt, args.wide_out);
        }
      };
      const size_t row_off = ((size_t)cur.bh * args.Tlen + grow) * D;
      if (MODE == MODE_DQ) {
        // dq = 2 / D_t x the sum, 32 columns per set
        uint32_t a0[32];
        float x[32];
        tmem_ld32(accu + set * 32, a0);
        tmem_wait_ld(a0);
        tc_fence_before();
        mbar_arrive(bar(BAR_OFREE));
        const float f = 2.f * inv_row;
#pragma unroll
        for (int c = 0; c < 32; ++c) x[c] = f * __uint_as_float(a0[c]);
        if constexpr (NS == 3) {
          const float back = grow < args.Tlen ? args.row_scale[(size_t)cur.bh * args.Tlen + grow] : 0.f;
#pragma unroll
          for (int c = 0; c < 32; ++c) x[c] *= back;
        }
        if (grow < args.Tlen) store32(args.out0 + row_off + set * 32, x);
      } else {
        // set 0: dk = r (2 u - r (k . 2 u) k);  set 1: dv = r dv~
        const unsigned char* kt = x1(ni & 1);
        auto krow = [&](int half, float (&kf)[32]) {
#pragma unroll
          for (int cix = 0; cix < 4; ++cix) {
            const uint4 raw = *reinterpret_cast<const uint4*>(kt + sw128_offset(rowl, half * 4 + cix));
            const uint32_t kw[4] = {raw.x, raw.y, raw.z, raw.w};
#pragma unroll
            for (int e = 0; e < 4; ++e) {
              const float2 f2 = unpack_bf16(kw[e]);
              kf[8 * cix + 2 * e] = f2.x;
              kf[8 * cix + 2 * e + 1] = f2.y;
            }
          }
        };
        float n2 = 0.f, dot = 0.f;
        uint32_t a0[32];
        float kf[32];
#pragma unroll 1
        for (int half = 0; half < 2; ++half) {
          krow(half, kf);
          tmem_ld32(accu + 64 + half * 32, a0);
          tmem_wait_ld(a0);
#pragma unroll
          for (int c = 0; c < 32; ++c) {
            n2 = fmaf(kf[c], kf[c], n2);
            dot = fmaf(kf[c], __uint_as_float(a0[c]), dot);
          }
        }
        const float r = inv_or_zero(n2);
        const float proj = r * dot;
        float back = 1.f;
        if constexpr (NS == 3) back = set == 0 && grow < args.Tlen ? args.row_scale[(size_t)cur.bh * args.Tlen + grow] : 1.f;
#pragma unroll 1
        for (int half = 0; half < 2; ++half) {
          float x[32];
          if (set == 0) krow(half, kf);
          tmem_ld32(accu + (set == 0 ? 64 : 0) + half * 32, a0);
          tmem_wait_ld(a0);
#pragma unroll
          for (int c = 0; c < 32; ++c)
            x[c] = set == 0 ? 2.f * r * (__uint_as_float(a0[c]) - proj * kf[c]) * back : r * __uint_as_float(a0[c]);
          if (grow < args.Tlen) store32((set == 0 ? args.out0 : args.out1) + row_off + half * 32, x);
        }
        tc_fence_before();
        mbar_arrive(bar(BAR_OFREE));
        mbar_arrive(bar(BAR_XEMPTY + (ni & 1)));
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

size_t align256(size_t n) { return (n + 255) / 256 * 256; }

// Pre-pass: one warp per 4 key rows (8 lanes x 16 bytes per row).  r = 1 / ||k||^2 (fp32).
__global__ void __launch_bounds__(256) bwd_rscale_kernel(const __nv_bfloat16* __restrict__ k, float* __restrict__ rk, size_t n_rows) {
  cudaTriggerProgrammaticLaunchCompletion();
  const size_t row = (size_t)blockIdx.x * 32 + (threadIdx.x >> 3);
  const int part = threadIdx.x & 7;
  if (row >= n_rows) return;
  const uint4 kraw = *reinterpret_cast<const uint4*>(k + row * D + part * 8);
  const uint32_t kw[4] = {kraw.x, kraw.y, kraw.z, kraw.w};
  float ss = 0.f;
#pragma unroll
  for (int e = 0; e < 4; ++e) {
    const float2 f = unpack_bf16(kw[e]);
    ss = fmaf(f.x, f.x, ss);
    ss = fmaf(f.y, f.y, ss);
  }
  ss += __shfl_xor_sync(0xffffffffu, ss, 1);
  ss += __shfl_xor_sync(0xffffffffu, ss, 2);
  ss += __shfl_xor_sync(0xffffffffu, ss, 4);
  if (part == 0) rk[row] = inv_or_zero(ss);
}

// The pre-pass of the three-term weights: also copies of the rows of k (blockIdx.y = 0) and q (1) scaled by the power of two that
// brings the largest entry to [1, 2), and that power; r is that of the scaled key.  An entry that the scaling takes below the
// smallest bf16 is 2^-126 of the row's largest.  Memory-bound, four rows per lane in flight.
constexpr int SCALE_ROWS = 4;
__global__ void __launch_bounds__(256) bwd_scale_kernel(const __nv_bfloat16* __restrict__ k, const __nv_bfloat16* __restrict__ q,
                                                        __nv_bfloat16* __restrict__ ks, __nv_bfloat16* __restrict__ qs, float* __restrict__ fk,
                                                        float* __restrict__ fq, float* __restrict__ rk, size_t n_rows) {
  cudaTriggerProgrammaticLaunchCompletion();
  const size_t row0 = (size_t)blockIdx.x * (32 * SCALE_ROWS) + (threadIdx.x >> 3);
  const int part = threadIdx.x & 7;
  const bool is_q = blockIdx.y != 0;
  const unsigned lanes = 0xFFu << (threadIdx.x & 24);       // the eight lanes of a row
  uint4 raw[SCALE_ROWS];
#pragma unroll
  for (int i = 0; i < SCALE_ROWS; ++i) {
    const size_t row = row0 + i * 32;
    raw[i] = make_uint4(0u, 0u, 0u, 0u);
    if (row < n_rows) raw[i] = *reinterpret_cast<const uint4*>((is_q ? q : k) + row * D + part * 8);
  }
#pragma unroll
  for (int i = 0; i < SCALE_ROWS; ++i) {
    const size_t row = row0 + i * 32;
    const uint32_t w[4] = {raw[i].x, raw[i].y, raw[i].z, raw[i].w};
    uint32_t top = 0;                                       // largest exponent field of the row
#pragma unroll
    for (int e = 0; e < 4; ++e) top = max(top, max(w[e] & 0x7F80u, (w[e] >> 16) & 0x7F80u));
#pragma unroll
    for (int off = 1; off < 8; off <<= 1) top = max(top, __shfl_xor_sync(lanes, top, off));
    const uint32_t ex = min(max(top >> 7, 1u), 253u);
    const float f = __uint_as_float((254u - ex) << 23);     // 2^(127 - ex)
    uint32_t s[4];
    float ss = 0.f;
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      const float2 x = unpack_bf16(w[e]);
      s[e] = pack_bf16(x.x * f, x.y * f);
      const float2 y = unpack_bf16(s[e]);
      ss = fmaf(y.x, y.x, ss);
      ss = fmaf(y.y, y.y, ss);
    }
#pragma unroll
    for (int off = 1; off < 8; off <<= 1) ss += __shfl_xor_sync(lanes, ss, off);
    if (row >= n_rows) continue;
    *reinterpret_cast<uint4*>((is_q ? qs : ks) + row * D + part * 8) = make_uint4(s[0], s[1], s[2], s[3]);
    if (part != 0) continue;
    (is_q ? fq : fk)[row] = f;
    if (!is_q) rk[row] = inv_or_zero(ss);
  }
}

template <int MODE, int G, int NS>
bool launch_bwd(const CUtensorMap& x1, const CUtensorMap& x2, const CUtensorMap& y1, const CUtensorMap& y2, const BArgs& a, LaunchCtx& ctx) {
  auto kern = tc_bwd_kernel<MODE, G, NS>;
  const int sms = sm_count();
  const long long n_items = (long long)a.BH * ((a.Tlen + MT - 1) / MT);
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(n_items < sms ? n_items : sms));   // persistent: one CTA per SM
  cfg.blockDim = dim3(Geo<MODE, G, NS>::NTHREADS);
  cfg.dynamicSmemBytes = SMEM_ALLOC;
  cfg.stream = ctx.stream;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  if (!allow_smem<tc_bwd_kernel<MODE, G, NS>>((int)SMEM_ALLOC) ||
      cudaLaunchKernelEx(&cfg, kern, x1, x2, y1, y2, a) != cudaSuccess) {
    cudaGetLastError();
    ctx.status = KATA_ERR_CUDA;
    return false;
  }
  ++ctx.launches;
  return true;
}

// Scratch: r, the row scalars, and with three terms the scaled rows and their powers of two.
struct BwdScratch {
  float* rk;                  // [BH][T]
  float* stats;               // [BH][T][2]
  __nv_bfloat16 *qs, *ks;     // [BH][T][64]
  float *fq, *fk;             // [BH][T]
};

// r, then dq and the row scalars, then dk and dv (which read the scalars)
template <int G, int NS>
void run_bwd(Problem p, const void* dout, void* dq, void* dk, void* dv, const BwdScratch& w, int* device_status, LaunchCtx& ctx) {
  const int BH = p.B * p.H;
  const size_t rows = (size_t)BH * p.T;
  constexpr int NT = Geo<MODE_DQ, G, NS>::NT;
  const __nv_bfloat16 *q = static_cast<const __nv_bfloat16*>(p.q), *k = static_cast<const __nv_bfloat16*>(p.k);
  const unsigned blocks = (unsigned)((rows + 31) / 32);
  if (NS == 3) {
    bwd_scale_kernel<<<dim3((blocks + SCALE_ROWS - 1) / SCALE_ROWS, 2), 256, 0, ctx.stream>>>(k, q, w.ks, w.qs, w.fk, w.fq, w.rk, rows);
    p.q = w.qs;
    p.k = w.ks;
  } else {
    bwd_rscale_kernel<<<blocks, 256, 0, ctx.stream>>>(k, w.rk, rows);
  }
  note_launch(ctx);
  CUtensorMap qf, gf, kf, vf, qs, gs, ks, vs;     // fixed tiles of 128 rows, streamed tiles of NT
  if (!make_tile_map(&qf, p.q, BH, p.T, MT) || !make_tile_map(&gf, dout, BH, p.T, MT) || !make_tile_map(&kf, p.k, BH, p.T, MT) ||
      !make_tile_map(&vf, p.v, BH, p.T, MT) || !make_tile_map(&qs, p.q, BH, p.T, NT) || !make_tile_map(&gs, dout, BH, p.T, NT) ||
      !make_tile_map(&ks, p.k, BH, p.T, NT) || !make_tile_map(&vs, p.v, BH, p.T, NT)) {
    ctx.status = KATA_ERR_CUDA;
    return;
  }
  const int wide = ((reinterpret_cast<uintptr_t>(dq) | reinterpret_cast<uintptr_t>(dk) | reinterpret_cast<uintptr_t>(dv)) & 31) == 0;
  BArgs a{static_cast<__nv_bfloat16*>(dq), nullptr, w.stats, w.rk, w.fq, device_status, wide, p.T, BH};
  if (!launch_bwd<MODE_DQ, G, NS>(qf, gf, ks, vs, a, ctx)) return;
  BArgs b{static_cast<__nv_bfloat16*>(dk), static_cast<__nv_bfloat16*>(dv), w.stats, w.rk, w.fk, device_status, wide, p.T, BH};
  launch_bwd<MODE_DKV, G, NS>(kf, vf, qs, gs, b, ctx);
}

}  // namespace

// workspace: r [BH][T] fp32, the row scalars [BH][T][2] fp32, and 128 bytes per row that are published but not used (k is read as
// it is)
size_t tc_bwd_workspace_bytes(const Problem& p) {
  const size_t rows = (size_t)p.B * p.H * p.T;
  return align256(rows * D * 2) + align256(rows * sizeof(float)) + align256(rows * 2 * sizeof(float));
}

void tc_bwd_quadratic(const Problem& p, const void* dout, void* dq, void* dk, void* dv, void* workspace, int* device_status,
                      LaunchCtx& ctx) {
  const size_t rows = (size_t)p.B * p.H * p.T;
  BwdScratch w{};
  w.rk = static_cast<float*>(workspace);
  w.stats = reinterpret_cast<float*>(static_cast<unsigned char*>(workspace) + align256(rows * sizeof(float)));
  if (p.groups == 1) run_bwd<1, 1>(p, dout, dq, dk, dv, w, device_status, ctx);
  else if (p.groups == 2) run_bwd<2, 1>(p, dout, dq, dk, dv, w, device_status, ctx);
  else run_bwd<4, 1>(p, dout, dq, dk, dv, w, device_status, ctx);
}

// The gradients with fp32 weights (three bf16 terms): kata_bwd_chunked on sequences short enough for the quadratic form.
size_t tc_bwd_exact_workspace_bytes(const Problem& p) {
  const size_t rows = (size_t)p.B * p.H * p.T;
  return 3 * align256(rows * sizeof(float)) + align256(rows * 2 * sizeof(float)) + 2 * align256(rows * D * 2);
}

void tc_bwd_exact(const Problem& p, const void* dout, void* dq, void* dk, void* dv, void* workspace, int* device_status, LaunchCtx& ctx) {
  const size_t rows = (size_t)p.B * p.H * p.T;
  unsigned char* w8 = static_cast<unsigned char*>(workspace);
  auto take = [&](size_t bytes) {
    unsigned char* at = w8;
    w8 += align256(bytes);
    return at;
  };
  BwdScratch w{};
  w.rk = reinterpret_cast<float*>(take(rows * sizeof(float)));
  w.stats = reinterpret_cast<float*>(take(rows * 2 * sizeof(float)));
  w.fq = reinterpret_cast<float*>(take(rows * sizeof(float)));
  w.fk = reinterpret_cast<float*>(take(rows * sizeof(float)));
  w.qs = reinterpret_cast<__nv_bfloat16*>(take(rows * D * 2));
  w.ks = reinterpret_cast<__nv_bfloat16*>(take(rows * D * 2));
  run_bwd<1, 3>(p, dout, dq, dk, dv, w, device_status, ctx);
}

}  // namespace kata
