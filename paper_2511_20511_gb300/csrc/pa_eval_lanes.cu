// pa_eval_lanes.cu -- launch shape of the lane-per-chromosome FP32 evaluation
// (pa_eval_lanes.cuh): which instances and counts it serves, how the columns
// are shared and the shared memory is laid out.
#include <algorithm>

#include "pa_eval_lanes.cuh"

namespace pa {

// Time (us) of a resident-table call by this kernel, to be held against
// small_eval_us (pa_fitness.cu).  Both kernels' times are staircases: what counts
// is the whole tiles of the busiest SM (m) and how often its blocks come round
// (`later` rounds beyond the first), so that a call changes sides several times
// as it grows (43 x 6, small calls' kernel / this one: 1.2 tiles per SM 16.3 /
// 21.9 us, 1.5: 23.0 / 21.8, 2.5: 27.8 / 31.7, 5: 50.5 / 49.2), and a line in the
// count alone sends calls to the slower one.  The terms: launch and fixed chain,
// buffers to fill, code to fetch (it grows with the columns), a unit's chain over
// the cells, gathers and decoding per tile, later rounds' chains.  Fitted to
// graph-replayed calls of 83 shapes (2 to 48 cells, 3 to 64 users) at 29 counts
// each: the kernel chosen is 0.8 % above the faster one in the mean (lines in the
// count: 2.5 %).  On 750 other calls of random shapes and counts: 0.4 %, and with
// lines 15 had been slower by 8 % and more than before there was a second kernel,
// up to 1.49 times.
static double lanes_us(const LanesArgs& a, int cols, int rounds, size_t smem, int64_t tiles,
                       int num_sms) {
  const int threads = (a.EW + a.NH) * 32;
  const int per_sm = std::max(1, std::min({(int)(kSmemPerSm / (smem + 1024 + 128)),
                                           65536 / (kLanesRegs * threads), 2048 / threads}));
  const double m = (double)((tiles + num_sms - 1) / num_sms), L = a.L, LK = L * a.K;
  const double later = (double)(((int64_t)m - 1) / per_sm);
  const double chain = 0.01 * rounds * L;
  return 4.45 + 1.64e-5 * smem + 1.47e-3 * cols * cols + 2.35 * chain +
         (2.74e-4 * L * LK + 5.8e-3 * LK) * m + 4.42 * later * chain;
}

// cudaErrorNotSupported where the kernel does not apply: a small call, or its
// buffers exceed shared memory.  Resident tables write fit[n]; column-tiled
// ones partial[n][ntile] (tiles_pay, pa_stream.cu).
cudaError_t launch_eval_lanes(pa_ctx* ctx, const uint8_t* pop, int64_t n, float* out,
                              cudaStream_t st) {
  const F32Tables& t = ctx->t32;
  if (t.streamed && !tiles_pay(ctx, n)) return cudaErrorNotSupported;
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
  a.L = L;
  a.K = K;
  if (!t.streamed) {
    // scalar rows of few cells: below 12 million gathered words never faster
    // (2 x 36, n = 8,728: 6.2 / 10.1 us; 7 x 20, n = 8,243: 7.7 / 8.8)
    if (t.vec == 1 && n * LK * L < 12000000) return cudaErrorNotSupported;
    const double us = lanes_us(a, cols, (units + a.EW - 1) / a.EW, b, tiles, ctx->num_sms);
    if (1.02 * us >= small_eval_us(ctx, n)) return cudaErrorNotSupported;
  }
  a.pop = pop;
  a.n = n;
  a.fit = out;
  a.tab = t.tab;
  a.own = t.own;
  a.bn = t.bn;
  a.err_flag = t.err_flag;
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
