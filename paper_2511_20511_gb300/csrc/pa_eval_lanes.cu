// pa_eval_lanes.cu -- launch shape of the lane-per-chromosome FP32 evaluation
// (pa_eval_lanes.cuh): which instances and counts it serves, how the columns
// are shared and the shared memory is laid out.
#include <algorithm>

#include "pa_eval_lanes.cuh"

namespace pa {

// Small calls stay with the kernels of fewer chromosomes per block
// (pa_fitness.cu, pa_stream.cu), which spread them over more SMs and start
// sooner.  Measured on GB300, those kernels against these:
//   37 x 13  n = 1024: 12.4 / 20.6 us   4096: 25.8 / 20.7   65536: 240 / 162
//   61 x 16 (column tiles)  n = 1024: 22.7 / 24.7 us   4096: 62.0 / 55.7
//   61 x 32 (column tiles, chunks)  n = 2^17: 2,853 / 2,348 us
// so the line lies where most SMs get a tile of 32 and the call gathers 12
// million table words.
bool lanes_applies(const pa_ctx* ctx, int64_t n) {
  const F32Tables& t = ctx->t32;
  const int64_t L = ctx->cfg.L, LK = L * ctx->cfg.K;
  const int64_t tiles = (n + kLanesTile - 1) / kLanesTile;
  if (n * LK * L < kLanesMinWords) return false;
  return t.streamed ? tiles * t.ntile >= ctx->num_sms : 5 * tiles >= 4 * ctx->num_sms;
}

// Tiles per SM from which it pays against the thread-per-(chromosome, pilot)
// kernel (K <= 16, L <= 24), x 10.  That kernel does no work for pad columns
// where L is a multiple of 4, and many pilots make this one's blocks few per SM.
// Measured, that kernel / this one:
//   19 x 10  n = 4096: 12.3 / 12.3 us   19,456: 22.0 / 18.6   48,000: 39.3 / 35.1
//   10 x 16  n = 13,000: 11.5 / 12.5    19,456: 14.6 / 12.5
//   16 x 16  n = 4096: 10.3 / 12.4      19,456: 20.8 / 24.8   80,000: 70.0 / 68.7
//   20 x 13  n = 4096: 10.3 / 13.8      19,456: 22.7 / 24.8   48,000: 47.3 / 43.3
//   24 x 4   n = 6144: 12.3 / 10.3      (K <= 8: never slower)
// With one block per SM (24 x 16) it stays behind: n = 300,000: 427 / 469 us.
static int64_t lanes_line(int L, int K) {
  return K <= 8 ? 8 : K > 12 && L % 4 == 0 ? 100 : 40;
}

// cudaErrorNotSupported where the kernel does not apply: a small call, or its
// buffers exceed shared memory.  Resident tables write fit[n]; column-tiled
// ones partial[n][ntile].
cudaError_t launch_eval_lanes(pa_ctx* ctx, const uint8_t* pop, int64_t n, float* out,
                              cudaStream_t st) {
  if (!lanes_applies(ctx, n)) return cudaErrorNotSupported;
  const F32Tables& t = ctx->t32;
  const int L = ctx->cfg.L, K = ctx->cfg.K, LK = L * K;
  const int64_t tiles = (n + kLanesTile - 1) / kLanesTile;
  LanesArgs a{};
  int cols;  // columns a block holds
  if (t.streamed) {
    a.ntile = t.ntile;
    a.JT = cols = t.JT;
    a.tab_floats = t.tile_floats;
  } else {
    a.ntile = 1;
    a.JT = cols = L;
    a.tab_floats = (((int64_t)LK * t.RS + 3) / 4) * 4;
  }
  if (cols > kLanesMaxNC) return cudaErrorNotSupported;
  a.NPR = (cols + 3) / 4 * 2;  // the column pairs of the table, pads included
  const int P = (cols + 1) / 2, JS = (P + kLanesMaxNP - 1) / kLanesMaxNP, W = (P + JS - 1) / JS;
  const size_t tile_bytes = (size_t)kLanesTile * LK;
  // the last piece decoded reads up to three rows and a word past the end
  a.xbytes = (int)(tile_bytes + ((3 * K + 16 + 15) & ~15));
  a.inv_words = ((L + 3) / 4) * K * kLanesTile;
  size_t b = 4 * (size_t)a.tab_floats;
  a.o_own = (int)b;
  b += 4 * (size_t)((LK + 3) & ~3);
  a.o_bn = (int)b;
  b += 4 * (size_t)((L + 3) & ~3);
  a.o_part = (int)b;
  b += 4 * (size_t)K * a.NPR * kLanesTile;
  a.o_sum = (int)b;
  b += 4 * kLanesTile;
  a.o_inv = (int)b;
  b += 8 * (size_t)a.inv_words;
  a.o_x = (int)b;
  a.xbufs = b + 2 * a.xbytes + 1024 <= (size_t)kSmemBudget ? 2 : 1;
  b += a.xbufs * (size_t)a.xbytes;
  if (b + 1024 > (size_t)kSmemBudget) return cudaErrorNotSupported;
  // 36 warps per SM (56 registers) in as many blocks as shared memory holds;
  // helper warps: their instructions per tile (decode: ~4 per byte, sum: ~4
  // per value, measured) with half again as margin, against one evaluation
  // warp's (a unit is ~17 per cell and pair of five columns and ~20 per pair),
  // since all warps of an SM get an equal part of its issue slots; evaluation
  // warps: the units (pilot, share) in equal rounds
  const int fit_blocks = std::max(1, (int)((size_t)kSmemBudget / (b + 1024)));
  if (!t.streamed && K <= 16 && L <= 24 &&
      (fit_blocks < 2 || 10 * tiles < lanes_line(L, K) * ctx->num_sms))
    return cudaErrorNotSupported;
  const int maxw = std::min(32, 36 / std::min(fit_blocks, 6));
  const int units = K * JS;
  const int unitw = L * (2 + 3 * W) + 22 * W, helpw = 4 * LK + 4 * K * a.NPR + 200;
  for (int nh = 2;; ++nh) {
    const int rounds = (units + maxw - nh - 1) / (maxw - nh);
    a.NH = nh;
    a.EW = (units + rounds - 1) / rounds;
    if (nh >= maxw - 1 || nh >= 8 || 2 * nh * rounds * unitw >= 3 * helpw) break;
  }
  // warps left over decode
  while (a.EW + a.NH < maxw && a.NH < 6 && a.NH >= 3) ++a.NH;
  a.pop = pop;
  a.n = n;
  a.fit = out;
  a.tab = t.tab;
  a.own = t.own;
  a.bn = t.bn;
  a.err_flag = t.err_flag;
  a.L = L;
  a.K = K;
  a.M = t.M;
  a.pc = t.pc;
  a.obj = ctx->cfg.objective;
  a.stall = ctx->test_stall;
  ctx->test_stall = 0;
  const bool fin = ctx->cfg.mode == PA_SINR_FINITE_M;
  LanesDispatch* go = t.vec == 2 ? (fin ? lanes_dispatch_fin2 : lanes_dispatch_asy2)
                                 : (fin ? lanes_dispatch_fin1 : lanes_dispatch_asy1);
  return go(cols, a, b, ctx->num_sms, tiles, st);
}

}  // namespace pa
