// Chunked KATA forward in fp32 on plain FMAs for rows of 16 or 32 entries (full lift, no state handed over): the states
// before chunks of 256 tokens, all chunks in parallel, then blocks of 32 or 64 queries over the state and the keys of their
// chunk.  Short sequences are one chunk: one launch, the quadratic form.
//   state_loc_kernel     S_loc = sum_t w psi(k_hat_t) [v_t, 1] over a chunk: thread = feature pair a <= b (w = 2 off the
//                        diagonal: the lift is symmetric), its DV + 1 sums in registers, rows broadcast from shared memory
//   state_prefix_kernel  running sum over the chunks, in order
//   attend_kernel        lane = one or two queries; the warps of a CTA share out the feature rows of the state and the tiles
//                        of 32 keys, rows broadcast from shared memory (16 bytes per load feed 8 FMAs), and add their
//                        numerators and normalisers in a fixed order at the end
// Few blocks: a cluster of CTAs shares the keys and the rows of one block, in tiles of 8 keys (2 heads x 512 tokens of 16
// entries: 32 blocks, whose warps walked 32 keys each, four to a scheduler, 8.9 us; as 128 CTAs 4.4).
// What bounds it: FMAs.  The walk over the chunks of a head by one CTA (kata_simt_chunked.cu) was a chain of 21 us per 64
// tokens: 2 heads x 512 tokens of 16 entries took 171 us, now 4.4; 16 x 16000 5378, now 242 (rows of 32: 12842, now 1197).
// Chunk length: at 16 entries a query costs 34 FMAs per key of its chunk and 2.3 k for the state, at 32 66 and 17 k.
#include <cooperative_groups.h>

#include <type_traits>

#include "kata_common.cuh"

namespace cg = cooperative_groups;

namespace kata {
namespace {

constexpr int CHUNK = 256;       // tokens per chunk

__host__ __device__ constexpr int n_features(int d) { return d * (d + 1) / 2; }
__host__ __device__ constexpr int state_stride(int dv) { return dv + 4; }       // [values | normaliser | 3 x padding]

__device__ __forceinline__ float4 ld4(const float* p) { return *reinterpret_cast<const float4*>(p); }

// rows [t0, t0 + n) of x (D entries each) into dst, normalised; rows from Tlen on are zero.  All threads of `nthr` (a multiple
// of D / 4, whole warps).
template <int D, bool NORM>
__device__ __forceinline__ void load_rows(const float* __restrict__ x, float* dst, int t0, int n, int Tlen, int thr, int nthr) {
  constexpr int PR = D / 4;      // lanes per row
  for (int i = thr; i < n * PR; i += nthr) {
    const int row = t0 + i / PR;
    float4 a = make_float4(0.f, 0.f, 0.f, 0.f);
    if (row < Tlen) a = ld4(x + (size_t)row * D + (i % PR) * 4);
    if (NORM) {
      float ss = a.x * a.x + a.y * a.y + a.z * a.z + a.w * a.w;
#pragma unroll
      for (int off = 1; off < PR; off <<= 1) ss += __shfl_xor_sync(0xffffffffu, ss, off);
      const float r = rsqrt_or_zero(ss);
      a.x *= r; a.y *= r; a.z *= r; a.w *= r;
    }
    *reinterpret_cast<float4*>(dst + i * 4) = a;
  }
}

template <int DK, int DV>
__global__ void __launch_bounds__((n_features(DK) + 31) / 32 * 32)
state_loc_kernel(const float* __restrict__ k, const float* __restrict__ v, float* __restrict__ S, int Tlen, int n_chunks) {
  constexpr int NF = n_features(DK), SP = state_stride(DV), NTHR = (NF + 31) / 32 * 32, TB = 64;
  __shared__ __align__(16) float ks[TB * DK], vs[TB * DV];
  const int c = blockIdx.x, bh = blockIdx.y, tid = threadIdx.x;
  int a = 0, rem = tid < NF ? tid : 0;
  while (rem >= DK - a) {
    rem -= DK - a;
    ++a;
  }
  const int b = a + rem;
  float acc[DV], den = 0.f;
#pragma unroll
  for (int i = 0; i < DV; ++i) acc[i] = 0.f;
  for (int t0 = c * CHUNK; t0 < (c + 1) * CHUNK; t0 += TB) {
    __syncthreads();
    load_rows<DK, true>(k + (size_t)bh * Tlen * DK, ks, t0, TB, Tlen, tid, NTHR);
    load_rows<DV, false>(v + (size_t)bh * Tlen * DV, vs, t0, TB, Tlen, tid, NTHR);
    __syncthreads();
#pragma unroll 4
    for (int t = 0; t < TB; ++t) {
      const float w = ks[t * DK + a] * ks[t * DK + b];
      den += w;
#pragma unroll
      for (int i = 0; i < DV; i += 4) {
        const float4 x = ld4(vs + t * DV + i);
        acc[i] = fmaf(w, x.x, acc[i]);
        acc[i + 1] = fmaf(w, x.y, acc[i + 1]);
        acc[i + 2] = fmaf(w, x.z, acc[i + 2]);
        acc[i + 3] = fmaf(w, x.w, acc[i + 3]);
      }
    }
  }
  if (tid >= NF) return;
  const float m = a == b ? 1.f : 2.f;
  float* dst = S + (((size_t)bh * n_chunks + c + 1) * NF + tid) * SP;
#pragma unroll
  for (int i = 0; i < DV; i += 4) *reinterpret_cast<float4*>(dst + i) = make_float4(m * acc[i], m * acc[i + 1], m * acc[i + 2], m * acc[i + 3]);
  *reinterpret_cast<float4*>(dst + DV) = make_float4(m * den, 0.f, 0.f, 0.f);
}

// S[1 .. n_chunks - 1] of every head: running sums; n4 = float4s per state, eight loads in flight
__global__ void __launch_bounds__(128) state_prefix_kernel(float4* __restrict__ S, int n4, int n_chunks) {
  cudaGridDependencySynchronize();
  const int i = blockIdx.x * 128 + threadIdx.x;
  if (i >= n4) return;
  float4* p = S + (size_t)blockIdx.y * n_chunks * n4 + i;
  float4 run = make_float4(0.f, 0.f, 0.f, 0.f);
  for (int c0 = 1; c0 < n_chunks; c0 += 8) {
    float4 x[8];
#pragma unroll
    for (int u = 0; u < 8; ++u)
      if (c0 + u < n_chunks) x[u] = p[(size_t)(c0 + u) * n4];
#pragma unroll
    for (int u = 0; u < 8; ++u)
      if (c0 + u < n_chunks) {
        run.x += x[u].x; run.y += x[u].y; run.z += x[u].z; run.w += x[u].w;
        p[(size_t)(c0 + u) * n4] = run;
      }
  }
}

template <int DK, int DV, int NW, int QPL, int CL> __host__ __device__ constexpr int attend_smem_floats() {
  const int tiles = 32 * QPL * DK + NW * 32 * (DK + DV), red = NW * (DV + 1) * 32 * QPL;
  return (tiles > red ? tiles : red) + (CL > 1 ? CL * (DV + 1) * 32 * QPL : 0);
}

// QPL queries per lane (a block is 32 QPL queries); NW warps share out its key tiles and state rows.  (One query per lane: two
// blocks per SM, rows of 32 with 132 registers lost the second and 16 heads x 512 tokens went from 27 to 33 us.)
// CL > 1: a cluster of CL CTAs does this for a block, in key tiles of TK, and adds its CTAs' sums in the shared memory of the
// first.
template <int DK, int DV, int NW, int QPL, int CL>
__global__ void __launch_bounds__(NW * 32, DK == 32 && DV == 32 && QPL == 1 ? 2 : 0) attend_kernel(const float* __restrict__ q, const float* __restrict__ k, const float* __restrict__ v,
                                                         float* __restrict__ out, const float* __restrict__ S, int Tlen, int chunk,
                                                         int n_chunks) {
  constexpr int NF = n_features(DK), SP = state_stride(DV), QB = 32 * QPL;
  constexpr int TK = CL > 1 ? 8 : 32;                      // keys per tile
  constexpr int GW = NW * CL;                              // warps that share a block
  extern __shared__ __align__(16) float smem[];
  float* sm = smem;
  float* qs = sm;                                          // [DK][QB]
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  float* kt = sm + QB * DK + warp * 32 * (DK + DV);        // this warp's tile: k_hat [32][DK], v [32][DV]
  float* vt = kt + 32 * DK;
  const int rank = CL > 1 ? (int)blockIdx.x % CL : 0, gw = rank * NW + warp;       // (a cluster is CL neighbours on x)
  const int q0 = ((int)gridDim.x / CL - 1 - (int)blockIdx.x / CL) * QB, bh = blockIdx.y;     // last blocks first
  const float* kh = k + (size_t)bh * Tlen * DK;
  const float* vh = v + (size_t)bh * Tlen * DV;
  const float* qh = q + (size_t)bh * Tlen * DK;
  if (CL > 1) asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory");     // this CTA has started
  if (S != nullptr) cudaGridDependencySynchronize();

  for (int i = tid; i < QB * DK; i += NW * 32) {
    const int row = i % QB, a = i / QB;
    qs[i] = q0 + row < Tlen ? qh[(size_t)(q0 + row) * DK + a] : 0.f;
  }
  __syncthreads();
  // normalised: the norm cancels in the ratio, but the weights of raw queries would leave the range of fp32 with its square
  float qr[QPL][DK], num[QPL][DV], den[QPL], rq[QPL];      // queries q0 + 32 u + lane
#pragma unroll
  for (int u = 0; u < QPL; ++u) {
    float ss[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
    for (int i = 0; i < DK; ++i) {
      qr[u][i] = qs[i * QB + 32 * u + lane];
      ss[i % 4] = fmaf(qr[u][i], qr[u][i], ss[i % 4]);
    }
    rq[u] = rsqrt_or_zero((ss[0] + ss[1]) + (ss[2] + ss[3]));
#pragma unroll
    for (int i = 0; i < DK; ++i) qr[u][i] *= rq[u];
    den[u] = 0.f;
#pragma unroll
    for (int i = 0; i < DV; ++i) num[u][i] = 0.f;
  }
  auto add = [&](const float* row, const float (&w)[QPL]) {
#pragma unroll
    for (int i = 0; i < DV; i += 4) {
      const float4 x = ld4(row + i);
#pragma unroll
      for (int u = 0; u < QPL; ++u) {
        num[u][i] = fmaf(w[u], x.x, num[u][i]);
        num[u][i + 1] = fmaf(w[u], x.y, num[u][i + 1]);
        num[u][i + 2] = fmaf(w[u], x.z, num[u][i + 2]);
        num[u][i + 3] = fmaf(w[u], x.w, num[u][i + 3]);
      }
    }
  };
  // ---- the state before the chunk ----
  const int c = q0 / chunk;
  if (c > 0) {
    const float* Sc = S + ((size_t)bh * n_chunks + c) * NF * SP;
    const int f0 = NF * gw / GW, f1 = NF * (gw + 1) / GW;
    int a = 0, rem = f0;
    while (rem >= DK - a) {
      rem -= DK - a;
      ++a;
    }
    int b = a + rem;
    float xa[QPL];                                         // (qs is as loaded: both factors of the norm go to x_a)
#pragma unroll
    for (int u = 0; u < QPL; ++u) xa[u] = qs[a * QB + 32 * u + lane] * rq[u] * rq[u];
    // sixteen rows at a time through this warp's tile buffer, the next sixteen on their way meanwhile
    constexpr int RB = 16, N4 = RB * SP / 4, PL = (N4 + 31) / 32;
    float4 pre[PL];
    auto fetch = [&](int f) {
      const int n4 = (f1 - f < RB ? f1 - f : RB) * SP / 4;
#pragma unroll
      for (int i = 0; i < PL; ++i)
        if (lane + 32 * i < n4) pre[i] = ld4(Sc + (size_t)f * SP + (lane + 32 * i) * 4);
    };
    fetch(f0);
    for (int fb = f0; fb < f1; fb += RB) {
      __syncwarp();
#pragma unroll
      for (int i = 0; i < PL; ++i)
        if (lane + 32 * i < N4) *reinterpret_cast<float4*>(kt + (lane + 32 * i) * 4) = pre[i];
      __syncwarp();
      if (fb + RB < f1) fetch(fb + RB);
      const int n = f1 - fb < RB ? f1 - fb : RB;
#pragma unroll 2
      for (int r = 0; r < n; ++r) {
        const float* row = kt + r * SP;
        const float z = row[DV];
        float w[QPL];
#pragma unroll
        for (int u = 0; u < QPL; ++u) {
          w[u] = xa[u] * qs[b * QB + 32 * u + lane];
          den[u] = fmaf(w[u], z, den[u]);
        }
        add(row, w);
        if (++b == DK) {
          b = ++a;
          if (a < DK) {
#pragma unroll
            for (int u = 0; u < QPL; ++u) xa[u] = qs[a * QB + 32 * u + lane] * rq[u] * rq[u];
          }
        }
      }
    }
  }
  // ---- the keys of the chunk ----
  const int k_end = min(q0 + QB, Tlen);
  for (int t0 = c * chunk + gw * TK; t0 < k_end; t0 += GW * TK) {
    __syncwarp();
    load_rows<DK, true>(kh, kt, t0, TK, Tlen, lane, 32);
    load_rows<DV, false>(vh, vt, t0, TK, Tlen, lane, 32);
    __syncwarp();
    const bool diag = t0 + TK - 1 > q0;
#pragma unroll 4
    for (int t = 0; t < TK; ++t) {
      float4 s4[QPL];                                      // (four partial sums: a chain of DK FMAs would set the pace)
#pragma unroll
      for (int u = 0; u < QPL; ++u) s4[u] = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
      for (int i = 0; i < DK; i += 4) {
        const float4 x = ld4(kt + t * DK + i);
#pragma unroll
        for (int u = 0; u < QPL; ++u) {
          s4[u].x = fmaf(qr[u][i], x.x, s4[u].x);
          s4[u].y = fmaf(qr[u][i + 1], x.y, s4[u].y);
          s4[u].z = fmaf(qr[u][i + 2], x.z, s4[u].z);
          s4[u].w = fmaf(qr[u][i + 3], x.w, s4[u].w);
        }
      }
      float w[QPL];
#pragma unroll
      for (int u = 0; u < QPL; ++u) {
        const float s = (s4[u].x + s4[u].y) + (s4[u].z + s4[u].w);
        w[u] = s * s;
        if (diag && t0 + t > q0 + 32 * u + lane) w[u] = 0.f;
        den[u] += w[u];
      }
      add(vt + t * DV, w);
    }
  }
  // ---- the warps' shares, in order ----
  __syncthreads();
  float* red = sm + warp * (DV + 1) * QB;                  // [warp][DV + 1][QB]
#pragma unroll
  for (int u = 0; u < QPL; ++u) {
#pragma unroll
    for (int i = 0; i < DV; ++i) red[i * QB + 32 * u + lane] = num[u][i];
    red[DV * QB + 32 * u + lane] = den[u];
  }
  __syncthreads();
  if constexpr (CL > 1) {
    // the CTA's sums to the first CTA of the cluster, which adds them in the order of the ranks
    float* all = sm + attend_smem_floats<DK, DV, NW, QPL, 1>();
    cg::cluster_group cluster = cg::this_cluster();
    asm volatile("barrier.cluster.wait.aligned;" ::: "memory");                         // ... as have the others
    float* dst = cluster.map_shared_rank(all, 0) + rank * (DV + 1) * QB;
    for (int i = tid; i < (DV + 1) * QB; i += NW * 32) {
      float x = 0.f;
#pragma unroll
      for (int w = 0; w < NW; ++w) x += sm[w * (DV + 1) * QB + i];
      dst[i] = x;
    }
    cluster.sync();
    if (rank != 0) return;
    sm = all;
  }
  constexpr int NSUM = CL > 1 ? CL : NW;
  const int row = tid % QB, part = tid / QB;               // four threads per query
  if (part >= 4) return;
  float dsum = 0.f;
#pragma unroll
  for (int w = 0; w < NSUM; ++w) dsum += sm[(w * (DV + 1) + DV) * QB + row];
  const float inv = dsum > 0.f ? 1.f / dsum : 0.f;
  if (q0 + row >= Tlen) return;
  constexpr int CPT = DV / 4;                              // columns per thread
  float* dst = out + ((size_t)bh * Tlen + q0 + row) * DV + part * CPT;
#pragma unroll
  for (int i = 0; i < CPT; i += 4) {
    float x[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
    for (int w = 0; w < NSUM; ++w)
#pragma unroll
      for (int e = 0; e < 4; ++e) x[e] += sm[(w * (DV + 1) + part * CPT + i + e) * QB + row];
    *reinterpret_cast<float4*>(dst + i) = make_float4(x[0] * inv, x[1] * inv, x[2] * inv, x[3] * inv);
  }
}

// measured, us, one chunk / chunks of 256: rows of 16, one head x 1024 tokens 6 / 22, 256 heads 349 / 247; rows of 32, one
// head x 1400 19 / 66, 128 heads x 1536 872 / 950
int one_chunk_tokens(const Problem& p) { return p.d_k == 32 ? 1536 : (long long)p.B * p.H * p.T <= 16384 ? 1024 : 512; }

template <int DK, int DV> void run(const Problem& p, float* S, LaunchCtx& ctx) {
  const int BH = p.B * p.H;
  const float *q = static_cast<const float*>(p.q), *k = static_cast<const float*>(p.k), *v = static_cast<const float*>(p.v);
  const bool states = p.T > one_chunk_tokens(p);
  const int chunk = states ? CHUNK : (p.T + 63) / 64 * 64, n_chunks = (p.T + chunk - 1) / chunk;
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.stream = ctx.stream;
  bool ok = true;
  if (states) {
    state_loc_kernel<DK, DV><<<dim3(n_chunks - 1, BH), (n_features(DK) + 31) / 32 * 32, 0, ctx.stream>>>(k, v, S, p.T, n_chunks);
    note_launch(ctx);
    const int n4 = n_features(DK) * state_stride(DV) / 4;
    cfg.gridDim = dim3((n4 + 127) / 128, BH);
    cfg.blockDim = dim3(128);
    cfg.numAttrs = 1;
    ok = cudaLaunchKernelEx(&cfg, state_prefix_kernel, reinterpret_cast<float4*>(S), n4, n_chunks) == cudaSuccess;
    ctx.launches += ok;
  }
  auto attend = [&](auto nw, auto qpl, auto cl) {
    constexpr int NW = decltype(nw)::value, QPL = decltype(qpl)::value, CL = decltype(cl)::value;
    constexpr int smem = attend_smem_floats<DK, DV, NW, QPL, CL>() * (int)sizeof(float);
    cfg.numAttrs = states ? 1 : 0;
    if (CL > 1) {
      attr[cfg.numAttrs].id = cudaLaunchAttributeClusterDimension;
      attr[cfg.numAttrs].val.clusterDim.x = CL;
      attr[cfg.numAttrs].val.clusterDim.y = attr[cfg.numAttrs].val.clusterDim.z = 1;
      ++cfg.numAttrs;
    }
    cfg.gridDim = dim3((p.T + 32 * QPL - 1) / (32 * QPL) * CL, BH);
    cfg.blockDim = dim3(NW * 32);
    cfg.dynamicSmemBytes = smem;
    return allow_smem<attend_kernel<DK, DV, NW, QPL, CL>>(smem) &&
           cudaLaunchKernelEx(&cfg, attend_kernel<DK, DV, NW, QPL, CL>, q, k, v, static_cast<float*>(p.out),
                              (const float*)(states ? S : nullptr), p.T, chunk, n_chunks) == cudaSuccess;
  };
  // Two queries per lane feed two FMAs per word loaded; where that makes fewer blocks than SMs, one query per lane and, if
  // the registers allow it, sixteen warps (2 heads x 512 tokens of 16 entries: 15.6 us of GPU time,
  // 13.4 with sixteen warps, 9.1 with one query per lane as well; 256 heads x 1024 tokens the other way round: 349 and 419).
  // Blocks that leave SMs idle have a cluster of CTAs each, as many as fit at once (a CTA of sixteen warps fills an SM, of eight
  // half of one), and where a block is long (1024 keys and more) two in any case.  Measured, us, CTAs per block 1 / 2 / 4 / 8: rows
  // of 16, two heads x 512 (32 blocks) 8.9 / 5.9 / 4.4 / 10.3, one x 1024 (32) 15.7 / 9.1 / 6.1 / 10.7, two x 1024 (64) 15.8 / 9.2 / 9.7 /
  // 17.7, eight x 512 (128) 9.2 / 10.6 / 15.1 / 31.3, four x 1024 (128) 15.8 / 14.2 / 18.0 / 31.5; rows of 32, one x 512 (16) 17.2 / 12.0 / 8.1 /
  // 7.4, one x 1024 (32) 31.0 / 20.1 / 12.3 / 10.5, two x 1024 (64) 31.0 / 20.6 / 16.9 / 17.7, eight x 1024 (256) 45.8 / 42.2 / 45.9 / 65.4.
  using std::integral_constant;
  const bool few = (long long)((p.T + 63) / 64) * BH <= sm_count();
  const long long blocks = (long long)((p.T + 31) / 32) * BH;
  constexpr bool wide = DK == 16 && DV == 16;
  constexpr integral_constant<int, wide ? 16 : 8> nw{};
  constexpr integral_constant<int, 1> one{};
  const long long slots = wide ? sm_count() : 2 * sm_count();
  if (!few) ok = ok && attend(integral_constant<int, 8>{}, integral_constant<int, 2>{}, one);
  else if (!wide && 8 * blocks <= slots) ok = ok && attend(nw, one, integral_constant<int, 8>{});
  else if (4 * blocks <= slots) ok = ok && attend(nw, one, integral_constant<int, 4>{});
  else if (2 * blocks <= slots || chunk >= 1024) ok = ok && attend(nw, one, integral_constant<int, 2>{});
  else ok = ok && attend(nw, one, one);
  if (!ok) {
    cudaGetLastError();
    ctx.status = KATA_ERR_CUDA;
    return;
  }
  ++ctx.launches;
}

}  // namespace

bool simt_attend_supported(const Problem& p) {
  return p.dtype == KATA_F32 && p.feature_order == 2 && p.groups == 1 && p.d_k <= 32 && p.d_v <= 32;
}

size_t simt_attend_workspace_bytes(const Problem& p) {
  if (p.T <= one_chunk_tokens(p)) return 0;
  return (size_t)p.B * p.H * ((p.T + CHUNK - 1) / CHUNK) * n_features(p.d_k) * state_stride(p.d_v) * sizeof(float);
}

void simt_attend(const Problem& p, float* ws, LaunchCtx& ctx) {
  if (p.d_k == 16) {
    if (p.d_v == 16) run<16, 16>(p, ws, ctx); else run<16, 32>(p, ws, ctx);
  } else {
    if (p.d_v == 16) run<32, 16>(p, ws, ctx); else run<32, 32>(p, ws, ctx);
  }
}

}  // namespace kata
