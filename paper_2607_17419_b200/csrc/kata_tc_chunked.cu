// Chunked (linear-state) KATA forward on the tensor cores, bf16: which launches make up each form.
// Sequential form (tc_chunked_states): the key scales, the states before the chunks (kata_tc_state.cu), the outputs
// (kata_tc_attend.cu); a short sequence is one chunk, the quadratic form alone.
// Scan forms and short calls with a state handed in or out (tc_chunked): the token-major streaming kernel
// (kata_tc_stream.cu); the scan forms run it over groups of 128-token tiles as reduce -> scan -> restart:
//   pass 1  every group but the last computes the state it adds (state-only mode: keys and values only)
//   pass 2  inclusive scan over the group states (scan_round_kernel, fp32 adds)
//   pass 3  every group starts from the prefix before it and writes its outputs
#include "kata_common.cuh"

namespace kata {

namespace {
size_t align256(size_t n) { return (n + 255) / 256 * 256; }

// Workspace of the chunk-state route: key scales, the states before the chunks, and with several segments their fp32 sums.
struct ChunkBuffers {
  size_t r, s, z, s_loc, z_loc, total;
};
ChunkBuffers chunk_buffers(const Problem& p, const StatePlan& plan, bool states) {
  const size_t BH = (size_t)p.B * p.H, slots = BH * plan.n_chunks, rows = (size_t)tc_state_rows(p);
  ChunkBuffers b{};
  b.r = 0;
  b.s = align256(BH * p.T * 4);
  b.z = b.s + (states ? align256(slots * rows * 64 * 2) : 0);
  b.s_loc = b.z + (states ? align256(slots * rows * 2) : 0);
  b.z_loc = b.s_loc + (states && plan.segments > 1 ? align256(slots * rows * 64 * 4) : 0);
  b.total = b.z_loc + (states && plan.segments > 1 ? align256(slots * rows * 4) : 0);
  return b;
}
}  // namespace

// Chunk length and segments.
// No state pointers and a short sequence: one chunk, the quadratic form alone.  Measured, us a call, quadratic / chunks, for 3, 16 and
// 128 heads:
//   full lift   T = 6000: 29 / 39, 65 / 92, 560 / 718     T = 7168: 34 / 47, 85 / 109, 766 / 833     T = 8192: 38 / 47, 107 / 131, 1022 / 1033
//               T = 10000: 44 / 50, 166 / 164, 1503 / 1187
//   two groups  T = 2500: 23 / 29, 29 / 46, 162 / 210     T = 3000: 25 / 29, 37 / 45, 234 / 243     T = 4096: 31 / 31, 50 / 55, 404 / 340
//   four groups T = 1500: 23 / 29, 23 / 33, 99 / 133      T = 2000: 27 / 29, 29 / 35, 155 / 142
//   rows of 32 entries (a third of the state)  T = 3000: 17 / 23, 24 / 35, 114 / 129     T = 3584: 19 / 23, 27 / 37, 150 / 176
//               T = 4096: 21 / 23, 30 / 37, 191 / 186     T = 4352: 22 / 25, 33 / 46, 201 / 213     T = 6000: 28 / 26, 56 / 51, 411 / 293
// The lines lie where the two were level with 128 heads (rows of 32: on both sides of 64 heads) when they were drawn.  The quadratic
// form has gained more since: the full lift's would lie near 8192 now.
// Chunks of 1024, one length for every map.  Shorter chunks write and read more state, longer ones have more key tiles, and the more keys
// reach a query through a bf16 state, the further its output is from 64 bits.  Measured, us, 512 / 768 / 1024:
//   full lift   16 x 131072 2005 / 2008 / 2007 (2048: 2138), 4 x 50001 292 / 267 / 246, 64 x 8192 490 / 488 / 475, 32 x 3001 with the state
//               out 103 / 102 / 105
//   two groups  4 x 50001 200 / 188 / 176, 16 x 32768 418 / 426 / 437, 128 x 4096 332 / 365 / 336
//   four groups 4 x 50001 148 / 153 / 151, 16 x 32768 359 / 368 / 391, 64 x 8192 299 / 328 / 350
// With feature groups and many heads 512 would be 1 to 15 % quicker and the outputs 1.0 to 2.2 % further from 64 bits (relative 2-norm, 512 /
// 1024: two groups 16 x 32768 2.60e-3 / 2.55e-3, 4 x 50001 2.45e-3 / 2.41e-3; four groups 16 x 32768 2.45e-3 / 2.41e-3, 64 x 8192 2.41e-3 /
// 2.38e-3; full lift 4 x 50001 2.95e-3 / 2.97e-3).
// Halved where even one chunk per CTA leaves SMs idle (3 heads x 2048 tokens with the state handed out: 37 -> 31 us).
StatePlan tc_chunk_plan(const Problem& p, bool state_in, bool state_out, bool small_scratch) {
  const int BH = p.B * p.H, slices = tc_state_rows(p) / 256;
  const int quad_tokens = tc_narrow(p) ? (BH < 64 ? 4352 : 3584) : p.groups == 1 ? 7168 : p.groups == 2 ? 3072 : 1536;
  StatePlan plan{};
  int L = 1024;
  if (!state_in && !state_out && p.T <= quad_tokens) L = (p.T + 255) / 256 * 256;
  else if (!small_scratch && (long long)BH * slices * ((p.T + L - 1) / L) < kPlanSMs) L = 512;
  plan.chunk_tokens = L;
  plan.n_chunks = (p.T + L - 1) / L;
  const int walk = state_out ? plan.n_chunks : plan.n_chunks - 1;
  plan.segments = kPlanSMs / (BH * slices);        // one CTA per SM
  if (plan.segments > walk) plan.segments = walk;
  if (plan.segments < 1) plan.segments = 1;
  plan.seg_chunks = walk > 0 ? (walk + plan.segments - 1) / plan.segments : 1;
  plan.segments = walk > 0 ? (walk + plan.seg_chunks - 1) / plan.seg_chunks : 1;
  return plan;
}

size_t tc_chunk_workspace_bytes(const Problem& p, const StatePlan& plan, bool state_in, bool state_out) {
  return chunk_buffers(p, plan, plan.n_chunks > 1 || state_in || state_out).total;
}

void tc_chunked_states(const Problem& p, const StatePlan& plan, void* workspace, int* device_status, const float* s_init,
                       const float* z_init, float* s_final, float* z_final, int state_layout, LaunchCtx& ctx) {
  const bool states = plan.n_chunks > 1 || s_init != nullptr || s_final != nullptr;
  const ChunkBuffers b = chunk_buffers(p, plan, states);
  unsigned char* w = static_cast<unsigned char*>(workspace);
  const bool exact_scales = p.groups > 1 || s_init != nullptr || s_final != nullptr;
  KeyScales r{};
  if (states || exact_scales) r.f32 = reinterpret_cast<float*>(w + b.r); else r.bf16 = reinterpret_cast<__nv_bfloat16*>(w + b.r);
  tc_rscale(p, r, ctx);
  AttendStates at{};
  at.exact_scales = exact_scales;
  if (states) {
    StateBuffers buf{};
    buf.s = reinterpret_cast<__nv_bfloat16*>(w + b.s);
    buf.z = reinterpret_cast<__nv_bfloat16*>(w + b.z);
    buf.s_loc = reinterpret_cast<float*>(w + b.s_loc);
    buf.z_loc = reinterpret_cast<float*>(w + b.z_loc);
    buf.s_init = s_init;
    buf.z_init = z_init;
    buf.s_final = s_final;
    buf.z_final = z_final;
    buf.layout = state_layout;
    if (ctx.status == KATA_OK) tc_states(p, r.f32, plan, buf, device_status, ctx);
    at.s = buf.s;
    at.z = buf.z;
    at.n_chunks = plan.n_chunks;
    at.chunk_tokens = plan.chunk_tokens;
    at.first_state = s_init != nullptr ? 0 : 1;
  }
  if (ctx.status == KATA_OK) tc_attend(p, r, at, device_status, ctx);
}

size_t tc_chunked_state_elems() { return tc_stream_state_elems(); }
int tc_chunked_slices() { return tc_stream_slices(); }

void tc_chunked(const Problem& p, const ScanPlan& plan, bool use_scan, float* ws, int* device_status,
                const float* s_init, const float* z_init, float* s_final, float* z_final, int state_layout,
                LaunchCtx& ctx) {
  if (!use_scan || plan.n_groups <= 1) {   // whole sequence in one pass
    if (s_final != nullptr || s_init != nullptr) {
      StreamIO io{};
      io.s_init = s_init;
      io.z_init = z_init;
      io.s_final = s_final;
      io.z_final = z_final;
      io.layout = state_layout;
      io.write_out = 1;
      tc_chunked_stream_export(p, device_status, io, ctx);
    } else {
      tc_chunked_stream(p, device_status, ctx);
    }
    return;
  }
  const int BH = p.B * p.H;
  const int NG = plan.n_groups;
  const size_t E = tc_chunked_state_elems();
  float* bufA = ws;
  float* bufB = ws + (size_t)BH * NG * E;
  StreamIO io{};
  io.layout = state_layout;
  io.n_groups = NG;
  io.tiles_per_group = plan.chunks_per_group * kChunk / tc_stream_tile();
  // pass 1: the states the groups add (the last group's is never needed)
  io.final_compact = bufA;
  io.write_out = 0;
  io.launch_groups = NG - 1;
  tc_chunked_stream_state(p, device_status, io, ctx);
  // pass 2
  const float* incl = scan_group_states(bufA, bufB, BH, NG, NG - 1, E, ctx);
  // pass 3
  io.init_compact = incl;
  io.final_compact = nullptr;
  io.write_out = 1;
  io.launch_groups = NG;
  tc_chunked_stream_restart(p, device_status, io, ctx);
}

}  // namespace kata
