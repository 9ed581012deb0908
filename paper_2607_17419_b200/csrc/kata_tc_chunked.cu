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
// No state pointers and a short sequence: one chunk, the quadratic form alone.  Per tile of 128 tokens and head the chunk
// states cost about 9 us of one SM to build and 7 to read (full lift), a key tile 0.55: the quadratic form wins until the
// average query sees about 29 key tiles.  Measured, us, quadratic / chunks of 1024, for 3, 16 and 128 heads:
//   full lift   T = 6000: 31 / 41, 75 / 92, 580 / 693     T = 7168: 35 / 51, 99 / 103, 784 / 835     T = 8192: 39 / 51, 123 / 123, 1172 / 936
//   two groups  T = 2500: 23 / 29, 37 / 47, 168 / 203     T = 3000: 26 / 29, 42 / 47, 236 / 227     T = 4096: 33 / 31, 53 / 58, 408 / 341
//   four groups T = 1500: 23 / 31, 24 / 35, 104 / 138     T = 2000: 29 / 31, 29 / 37, 166 / 147
//   rows of 32 entries (a third of the state)  T = 3000: 19 / 25, 28 / 41, 139 / 153     T = 4096: 25 / 26, 35 / 41, 232 / 211     T = 6000: 32 / 28, 67 / 61, 498 / 321
//   (few heads, whose blocks split the keys between the halves of a CTA, would take the quadratic form further: 3 heads up to
//   10000 tokens 45 / 53; the line is one for all heads)
// Chunks of 1024: 16 heads x 131072 tokens 2.08 ms; 768: 2.10, 512: 2.17, 2048 about 2.3 (shorter chunks write and read more state, longer
// ones have more key tiles).  One length for every map; measured, us, 512 / 768 / 1024: full lift 4 x 50001 313 / 276 / 249,
// 64 x 8192 540 / 523 / 508, 32 x 3001 with the state 117 / 111 / 111; two groups 4 x 50001 222 / 201 / 183, 16 x 32768
// 462 / 452 / 456, 128 x 4096 350 / 370 / 342; four groups 4 x 50001 166 / 166 / 160, 16 x 32768 378 / 373 / 395, 64 x 8192
// 334 / 354 / 373 (there 512 would be quicker).  Halved where even one chunk per CTA leaves SMs idle (3 heads x 2048 tokens with the state
// handed out: 43 -> 38 us).
StatePlan tc_chunk_plan(const Problem& p, bool state_in, bool state_out, bool small_scratch) {
  const int BH = p.B * p.H, slices = tc_state_rows(p) / 256;
  const int quad_tokens = tc_narrow(p) ? (BH < 64 ? 4352 : 3584) : p.groups == 1 ? 7168 : p.groups == 2 ? 3072 : 1536;
  StatePlan plan{};
  int L = 1024;
  if (!state_in && !state_out && p.T <= quad_tokens) L = (p.T + 255) / 256 * 256;
  else if (!small_scratch && (long long)BH * slices * ((p.T + L - 1) / L) < 148) L = 512;
  plan.chunk_tokens = L;
  plan.n_chunks = (p.T + L - 1) / L;
  const int walk = state_out ? plan.n_chunks : plan.n_chunks - 1;
  plan.segments = 148 / (BH * slices);        // one CTA per SM
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
