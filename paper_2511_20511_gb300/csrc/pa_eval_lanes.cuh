// pa_eval_lanes.cuh -- throughput form of the FP32 population evaluation
// (paper Sec. 3.2, Eq. 3-6): a lane per chromosome, a warp per pilot.
//
// A tile is 32 chromosomes.  Lane c of every warp works on chromosome c of
// the tile; an evaluation warp takes a unit = (pilot p, share h of the BS
// columns), walks the L cells and adds, per cell, the table row of the user
// that holds p -- the sums, their order and the SINR steps are those of
// eval_pilot_f32, so every per-(pilot, column pair) value and every fitness
// is bit for bit what the other FP32 kernels compute.
//
// What bounds it is the shared-memory data path: 32 words per clock and SM.
// The gathers themselves need L^2 K words per chromosome (113 wavefronts for
// 19 x 10); the layout keeps everything else small beside them:
//   * table rows: 32 lanes read at most K distinct rows of one cell, whose
//     odd pitch puts them in distinct banks (equal rows broadcast); the column
//     count is a template parameter, so that columns past L are not read and
//     nothing is tested per cell;
//   * the decoded inverse INV[(l/4)*K + p][c] holds the users of four cells
//     per word: one conflict-free load per four cells (against a byte load
//     per cell), and decoding scatters bytes into the lane's own bank, so
//     its stores never conflict whatever the permutation;
//   * per-(pilot, pair) values PART[p*NPR + q][c]: conflict-free both ways;
//     the member sum runs the fixed 32-lane tree inside a lane (no shuffles,
//     which share the data path).
// A unit holds at most six column pairs, so that 36 warps of 56 registers fit
// an SM, and keeps its code short (with decoding in every warp's path the
// instruction cache missed: 720 us against 571 below).  Rows and own gains are
// addressed by one dp4a each, columns are processed as f32x2 pairs (637 -> 406
// warp instructions per chromosome).
// Helper warps decode tile i+1 and sum tile i-1 while the evaluation warps
// gather tile i, so the data path stays busy through those phases; warps wait
// for one another only through mbarriers (a tile of slack), not through block
// barriers.  Chromosome bytes arrive by one bulk copy per tile, the table by
// bulk copies at the start.
// Measured (GB300, finite-M SINR): 2^20 chromosomes of 19 x 10 in 571 us, 6,630
// Gword/s of gathers, the data path 85 % busy with 145 wavefronts per chromosome
// (the kernel with a thread per (chromosome, pilot): 739 us, 177 wavefronts);
// 65,536 of 37 x 16 in 194 us (370 us); 100,003 of 19 x 24 in 141 us (224 us); 65,536
// of 61 x 12, column tiles, in 408 us (618 us).
#pragma once

#include <algorithm>
#include <type_traits>
#include <utility>

#include "pa_eval_device.cuh"

namespace pa {

constexpr int kLanesRegs = 56;        // 36 warps per SM
constexpr int kLanesMaxNP = 6;        // column pairs per unit at most
constexpr int kLanesMaxNC = 48;       // columns per block at most

struct LanesArgs {
  const uint8_t* pop;
  int64_t n;
  float* fit;       // [n], or partial sums [n][ntile] of the column tiles
  const float* tab; // column tile t at tab + t * tab_floats
  const float* own;
  const float* bn;
  int* err_flag;    // null: no bulk copies
  int L, K;
  int ntile, JT;    // column tiles (1: the whole table) and their width
  int NPR;          // column pairs per pilot in PART
  int EW, NH;       // evaluation and helper warps
  int xbufs;        // chromosome buffers (1 or 2)
  int xbytes;       // bytes of one
  int o_own, o_bn, o_part, o_sum, o_inv, o_x;  // shared-memory offsets
  int inv_words;    // words of one inverse buffer
  int64_t tab_floats;
  float M, pc;
  int obj;
  int stall;        // testing: announce the chromosome copies, never issue them
};

// The launch of one variant (columns NC per block; FINITE_M or not, float2
// or scalar table rows), one translation unit each: pa_eval_lanes_*.cu.
using LanesDispatch = cudaError_t(int NC, const LanesArgs& a, size_t smem, int num_sms,
                                  int64_t tiles, cudaStream_t st);
LanesDispatch lanes_dispatch_fin2, lanes_dispatch_fin1, lanes_dispatch_asy2, lanes_dispatch_asy1;

namespace {

__device__ __forceinline__ void bar_sync(int id, int n) {
  asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(n) : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint32_t mb) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(mb) : "memory");
}

__device__ __forceinline__ uint2 lds64(uint32_t addr) {
  uint2 v;
  asm volatile("ld.shared.v2.u32 {%0, %1}, [%2];" : "=r"(v.x), "=r"(v.y) : "r"(addr));
  return v;
}
__device__ __forceinline__ void sts8(uint32_t addr, uint32_t v) {
  asm volatile("st.shared.u8 [%0], %1;" ::"r"(addr), "r"(v) : "memory");
}

// Users k .. k+3 (the first n of them real) of four rows, a word each: byte b
// of v[s] is the pilot of user k + b in row s; dst: shared address of lane c's
// byte of the quad's word for pilot 0.  A valid row's bytes are below K: one
// test for all sixteen (bytes with the top bit set, or reaching it when 128 - K
// is added), byte by byte otherwise.  dp4a with one non-zero selector byte is a
// byte's extraction, scaling by the 128 bytes between pilots and base addition
// in one instruction.
__device__ __forceinline__ void lanes_put(uint32_t (&v)[4], uint32_t dst, uint32_t k, int n,
                                          int K) {
  const uint32_t lim = (uint32_t)(128 - K) * 0x01010101u;
  if (n < 4) {
    const uint32_t keep = (1u << (8 * n)) - 1u;
#pragma unroll
    for (int s = 0; s < 4; ++s) v[s] &= keep;
  }
  uint32_t odd = 0;
#pragma unroll
  for (int s = 0; s < 4; ++s) odd |= v[s] | (v[s] + lim);
  if ((odd & 0x80808080u) == 0) {
#pragma unroll
    for (int b = 0; b < 4; ++b)
      if (b < n) {
#pragma unroll
        for (int s = 0; s < 4; ++s) sts8(__dp4a(v[s], 128u << (8 * b), dst) + s, k + b);
      }
  } else {
    for (int b = 0; b < 4 && b < n; ++b)
#pragma unroll
      for (int s = 0; s < 4; ++s) {
        const uint32_t p = (v[s] >> (8 * b)) & 0xffu;
        if (p < (uint32_t)K) sts8(dst + p * 128 + s, k + b);
      }
  }
}

// Sixteen users k0 .. k0+15 (the first nb of them real) of four rows K bytes
// apart, row: shared address of user k0's byte of the first.
__device__ __forceinline__ void lanes_decode16(uint32_t row, uint32_t dst, int k0, int nb, int K) {
  constexpr int R = 4;
  auto put = [&](uint32_t (&v)[R], int w) {
    lanes_put(v, dst, (uint32_t)(k0 + 4 * w), nb - 4 * w, K);
  };
  if (K % 8 == 0) {  // 8-byte rows: L*K/8 odd keeps a half-warp's loads apart
#pragma unroll
    for (int h = 0; h < 2; ++h)
      if (8 * h < nb) {
        uint32_t v[2][R];
#pragma unroll
        for (int s = 0; s < R; ++s) {
          const uint2 w = lds64(row + s * K + 8 * h);
          v[0][s] = w.x;
          v[1][s] = w.y;
        }
        put(v[0], 2 * h);
        put(v[1], 2 * h + 1);
      }
  } else {  // any alignment: words realigned by a funnel shift
    uint32_t a[R], sh[R], w0[R], v[R];
#pragma unroll
    for (int s = 0; s < R; ++s) {
      a[s] = (row + s * K) & ~3u;
      sh[s] = 8 * (row + s * K);  // (taken modulo 32)
      w0[s] = lds32(a[s]);
    }
#pragma unroll
    for (int w = 0; w < 4; ++w)
      if (4 * w < nb) {
#pragma unroll
        for (int s = 0; s < R; ++s) {
          const uint32_t w1 = lds32(a[s] + 4 * w + 4);
          v[s] = __funnelshift_r(w0[s], w1, sh[s]);
          w0[s] = w1;
        }
        put(v, w);
      }
  }
}

// Lane c's chromosome (x: shared address of its L*K bytes) into the inverse:
// byte l&3 of word INV[((l>>2)*K + p)*32 + c] = k where row l gives pilot p to
// user k (inv: shared address of INV + c).  Pilots >= K are skipped (the byte
// keeps an earlier user, always < K).  Decoder h of nh takes every nh-th
// piece of four rows and sixteen users; rows past L in the last piece are the
// bytes that follow (the next chromosome's first rows, or the buffer's pad),
// and land in bytes that no one reads.
__device__ __noinline__ void lanes_decode(uint32_t x, uint32_t inv, int L, int K, int h, int nh) {
  const int nch = (K + 15) >> 4, items = ((L + 3) >> 2) * nch;
  for (int it = h; it < items; it += nh) {
    const int g = it / nch, k0 = 16 * (it - g * nch);
    const uint32_t row = x + 4 * g * K + k0, dst = inv + g * K * 128;
    const int nb = min(16, K - k0);
    lanes_decode16(row, dst, k0, nb, K);
  }
}

// Shared addresses a unit reads (lane c's column of the inverse, the tables).
struct LanesView {
  uint32_t T, OWN, BN, inv;
  int L, K, jb, jn;  // jb: BS of the block's column 0; jn: its real columns
  f32x2 M, pc;
};

// One unit: columns C0 .. C0+NC-1 of the block for one pilot and lane c
// (v.inv: INV + p*32 + c).  With TILED only the block's first jn columns are
// real.  Writes part[q*32] for the unit's pairs after ready() (the previous
// tile's values have been summed).
template <int C0, int NC, int RS, int VEC, bool FIN, bool TILED, typename Ready>
__device__ __forceinline__ void lanes_unit(const LanesView& v, bool minobj, float* part,
                                           Ready ready) {
  constexpr int NP = (NC + 1) / 2;
  constexpr bool ODD = (NC & 1) != 0;
  const int L = v.L, K = v.K;
  f32x2 acc2[NP];
  f32x2 acc1[FIN ? NP : 1];
#pragma unroll
  for (int q = 0; q < NP; ++q) {
    acc2[q] = 0;
    if (FIN) acc1[q] = 0;
  }
  float tail2 = 0.f, tail1 = 0.f;  // an odd last column's sums
  auto cell = [&](uint32_t row) {
#pragma unroll
    for (int q = 0; q < NP; ++q) {
      if (ODD && q == NP - 1) {
        const float x = lds_f(row + 8 * q);
        tail2 = __fmaf_rn(x, x, tail2);
        if (FIN) tail1 = __fadd_rn(tail1, x);
      } else {
        const f32x2 x =
            VEC == 2 ? lds_x2(row + 8 * q) : pk(lds_f(row + 8 * q), lds_f(row + 8 * q + 4));
        acc2[q] = fma2(x, x, acc2[q]);
        if (FIN) acc1[q] = add2(acc1[q], x);
      }
    }
  };
  // row of user u (byte s of w): base + u * RS * 4 by one dp4a (RS * 4 < 256)
  uint32_t Tl = v.T + 4 * C0;
  const uint32_t KRS = 4u * K * RS, KW = 128u * K;
  uint32_t iw = v.inv;
  int l = 0;
  for (; l + 4 <= L; l += 4) {
    const uint32_t w = lds32(iw);
    iw += KW;
#pragma unroll
    for (int s = 0; s < 4; ++s) {
      cell(__dp4a(w, (uint32_t)(4 * RS) << (8 * s), Tl));
      Tl += KRS;
    }
  }
  if (l < L) {
    uint32_t w = lds32(iw);
    for (; l < L; ++l, w >>= 8) {
      cell(__dp4a(w, (uint32_t)(4 * RS), Tl));
      Tl += KRS;
    }
  }
  if (ODD) {
    acc2[NP - 1] = pk(tail2, 0.f);
    if (FIN) acc1[NP - 1] = pk(tail1, 0.f);
  }
  ready();
  auto finish = [&](auto mobj) {
    constexpr bool mo = decltype(mobj)::value;
    uint32_t uw = 0;
    uint32_t own = v.OWN + 4u * (v.jb + C0) * K;
    iw = v.inv + (uint32_t)((v.jb + C0) >> 2) * KW;
    const uint32_t bn = v.BN + 4u * (v.jb + C0);
#pragma unroll
    for (int q = 0; q < NP; ++q) {
      float ps = pair_init(mo);
      const int c0 = C0 + 2 * q;  // (jb is a multiple of four)
      if (!TILED || c0 < v.jn) {
        if (q == 0 || (c0 & 3) == 0) {  // users of four cells
          uw = lds32(iw);
          iw += KW;
        }
        const bool two = 2 * q + 1 < NC;
        const f32x2 b =
            pk(lds_f(__dp4a(uw, 4u << (8 * (c0 & 3)), own)),
               two ? lds_f(__dp4a(uw, 4u << (8 * (c0 & 3) + 8), own + 4 * K)) : 1.f);
        own += 8 * K;
        const float2 x = se_pair_f32<FIN, mo>(acc2[q], FIN ? acc1[q] : 0, b,
                                              FIN ? lds_x2(bn + 8 * q) : 0, v.M, v.pc);
        ps = x.x;
        if (two && (!TILED || c0 + 1 < v.jn)) ps = pair_add(ps, x.y, mo);
      }
      part[q * 32] = ps;
    }
  };
  if (minobj)
    finish(std::true_type{});
  else
    finish(std::false_type{});
}

// Member values of a tile from PART by the first two helper warps: the same
// additions in the same tree as member_sum (lane i of that tree adds entries
// i, i+32, ...; then pairs at distance 16, 8, 4, 2, 1): helper h takes the
// tree's lanes i with i % 2 == h in registers, the last level joins the two.
template <bool MO>
__device__ __forceinline__ float lanes_sum_half(const float* PART, int total, int h) {
  float s[16];
#pragma unroll
  for (int k = 0; k < 16; ++k) s[k] = pair_init(MO);
  int r = h;
  for (; r + 30 < total; r += 32) {
#pragma unroll
    for (int k = 0; k < 16; ++k) s[k] = pair_add(s[k], PART[(r + 2 * k) * 32], MO);
  }
#pragma unroll
  for (int k = 0; k < 16; ++k)
    if (r + 2 * k < total) s[k] = pair_add(s[k], PART[(r + 2 * k) * 32], MO);
#pragma unroll
  for (int w = 8; w > 0; w >>= 1)
#pragma unroll
    for (int k = 0; k < w; ++k) s[k] = pair_add(s[k], s[k + w], MO);
  return s[0];
}

__device__ __noinline__ void lanes_sum(const float* PART, int total, float* SUMX, int h,
                                          int lane, bool mo, float* out, int64_t stride,
                                          int nvalid) {
  const float s = mo ? lanes_sum_half<true>(PART + lane, total, h)
                     : lanes_sum_half<false>(PART + lane, total, h);
  if (h == 1) SUMX[lane] = s;
  bar_sync(2, 64);
  if (h == 0 && lane < nvalid) out[lane * stride] = pair_add(s, SUMX[lane], mo);
}

// NC: columns of a block (the instance's L, or the width of a column tile
// -- widths 4, 8 and 16, which then serve any L).
template <int NC>
struct LanesShape {
  static constexpr bool kTiled = NC == 4 || NC == 8 || NC == 16;
  static constexpr int kP = (NC + 1) / 2;                          // real pairs
  static constexpr int kJS = (kP + kLanesMaxNP - 1) / kLanesMaxNP;  // column shares
  static constexpr int kW = 2 * ((kP + kJS - 1) / kJS);            // columns of all but the last
  static constexpr int kNJ = (NC + 3) / 4 * 4;
};

// Share h of pilot p: the unit whose first column is known at compile time.
template <int H, int NC, int RS, int VEC, bool FIN, typename Ready>
__device__ __forceinline__ void lanes_share(LanesView& v, int h, int p, bool minobj, float* part,
                                            Ready ready) {
  using Sh = LanesShape<NC>;
  if constexpr (H < Sh::kJS) {
    if (h == H) {
      constexpr int C0 = H * Sh::kW, N = H == Sh::kJS - 1 ? NC - C0 : Sh::kW;
      v.inv += p * 128;
      lanes_unit<C0, N, RS, VEC, FIN, Sh::kTiled>(v, minobj, part + C0 / 2 * 32, ready);
      v.inv -= p * 128;
    } else {
      lanes_share<H + 1, NC, RS, VEC, FIN>(v, h, p, minobj, part, ready);
    }
  }
}

template <int NC, int VEC, bool FIN>
__global__ void __maxnreg__(kLanesRegs) k_eval_f32_lanes(const LanesArgs a) {
  extern __shared__ __align__(128) unsigned char smem[];
  // [0, 1] chromosome buffers, [2] table: bulk copies;
  // [3, 4] a tile's inverse is decoded (decoders), [5, 6] its values are
  // written and its inverse is free (evaluation warps), by tile parity;
  // [7] its values are summed (the two sum warps)
  __shared__ __align__(8) uint64_t mbar[8];
  using Sh = LanesShape<NC>;
  constexpr int RS = Sh::kNJ + (VEC == 2 ? 2 : 1);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nthr = blockDim.x;
  const int L = Sh::kTiled ? a.L : NC, K = a.K, LK = L * K, EW = a.EW;
  // helper warps: the first two sum; all decode, or the others alone when there
  // are enough of them
  const int D0 = a.NH >= 4 ? 2 : 0, ND = a.NH - D0;
  float* T = reinterpret_cast<float*>(smem);
  float* OWN = reinterpret_cast<float*>(smem + a.o_own);
  float* BN = reinterpret_cast<float*>(smem + a.o_bn);
  float* PART = reinterpret_cast<float*>(smem + a.o_part);
  float* SUMX = reinterpret_cast<float*>(smem + a.o_sum);
  uint32_t* INV = reinterpret_cast<uint32_t*>(smem + a.o_inv);
  uint8_t* X = smem + a.o_x;
  const int t = blockIdx.x % a.ntile;
  const int64_t b = blockIdx.x / a.ntile, nb = gridDim.x / a.ntile;
  const int jb = t * a.JT;                          // first BS of the block's columns
  const int jn = min(L - jb, a.JT);                 // its real columns
  const int64_t tiles = (a.n + kLanesTile - 1) / kLanesTile;
  const int tile_bytes = kLanesTile * LK;           // a multiple of 32
  const bool bulk = a.err_flag != nullptr && (reinterpret_cast<uintptr_t>(a.pop) & 15) == 0;
  const bool mo = a.obj != 0;
  const uint32_t mb0 = smem_u32(&mbar[0]);
  auto bytes_of = [&](int64_t tile) {
    return (int)min((int64_t)tile_bytes, (a.n - tile * kLanesTile) * LK);
  };
  auto issue = [&](int64_t tile, int buf) {  // one thread: the tile's whole 16-byte units
    const uint32_t by = (uint32_t)bytes_of(tile) & ~15u, mb = mb0 + 8 * buf;
    mbar_expect_tx(mb, by);
    if (by && !a.stall)
      bulk_g2s(smem_u32(X + buf * a.xbytes), a.pop + tile * (int64_t)tile_bytes, by, mb);
  };
  if (tid == 0) {
    for (int i = 0; i < 3; ++i) mbar_init(mb0 + 8 * i, 1);
    for (int i = 0; i < 2; ++i) {
      mbar_init(mb0 + 8 * (3 + i), ND);
      mbar_init(mb0 + 8 * (5 + i), EW);
    }
    mbar_init(mb0 + 8 * 7, 2);
  }
  __syncthreads();
  const float* tab = a.tab + t * a.tab_floats;
  if (bulk) {
    if (tid == 0) {
      for (int i = 0; i < a.xbufs; ++i)
        if (b + i * nb < tiles) issue(b + i * nb, i);
      const uint32_t bytes = (uint32_t)(a.tab_floats * 4), mb = mb0 + 8 * 2;
      mbar_expect_tx(mb, bytes);
      constexpr uint32_t kChunk = 32768;
      for (uint32_t off = 0; off < bytes; off += kChunk)
        bulk_g2s(smem_u32(T) + off, reinterpret_cast<const char*>(tab) + off,
                 min(kChunk, bytes - off), mb);
    }
  } else {
    const float4* s4 = reinterpret_cast<const float4*>(tab);
    for (int i = tid; i < (int)(a.tab_floats / 4); i += nthr)
      reinterpret_cast<float4*>(T)[i] = __ldg(s4 + i);
  }
  for (int i = tid; i < LK; i += nthr) OWN[i] = __ldg(a.own + i);
  for (int i = tid; i < ((L + 3) & ~3); i += nthr) BN[i] = FIN && i < L ? __ldg(a.bn + i) : 0.f;
  for (int i = tid; i < 2 * a.inv_words; i += nthr) INV[i] = 0;  // users stay < K
  // the pads behind the chromosomes read as pilot 0
  for (int i = tid; i < a.xbytes - tile_bytes; i += nthr)
    for (int k = 0; k < a.xbufs; ++k) X[k * a.xbytes + tile_bytes + i] = 0;
  // pairs past the last column are never written again: neutral in the sums
  for (int i = tid; i < K * a.NPR * 32; i += nthr) PART[i] = pair_init(mo);
  __syncthreads();

  // A wait that gives up (about a second) sets the error flag; the warp then
  // waits for no more copies and the block runs its tiles to the end with
  // what its buffers hold (valid users by construction, results unspecified).
  int late = 0;  // 1: waits for no more copies, 2: nor for the block's own warps
  auto wait_copy = [&](int m, uint32_t ph) {
    if (!bulk || late || mbar_wait(mb0 + 8 * m, ph)) return;
    if (lane == 0) atomicExch(a.err_flag, 1);
    mbar_wait(mb0 + 8 * m, ph);  // a bounded chance to land before its buffer is left
    late = 1;
  };
  // The block's own warps always arrive, a late one after two of its waits:
  // the bound here is a net, several times that.  A late warp waits for the
  // others as before: one that ran ahead would complete phases that they have
  // not seen, and they would sit their whole bound out (a call whose copies
  // never come returned after 9.7 s that way).
  auto wait_warps = [&](int m, int i) {
    for (int k = 0; k < 8 && late < 2; ++k)
      if (mbar_wait(mb0 + 8 * m, (uint32_t)i & 1)) return;
    if (lane == 0 && late < 2 && a.err_flag) atomicExch(a.err_flag, 1);
    late = 2;
  };
  auto arrive = [&](int m) {
    __syncwarp();
    if (lane == 0) mbar_arrive(mb0 + 8 * m);
  };

  if (warp < EW) {
    // ---- evaluation warps: the units of each tile in turn
    LanesView view{smem_u32(T), smem_u32(OWN), smem_u32(BN), 0, L, K, jb, jn,
                   pk(a.M, a.M), pk(a.pc, a.pc)};
    const int units = K * Sh::kJS;
    wait_copy(2, 0);
    int i = 0;
    for (int64_t tile = b; tile < tiles; tile += nb, ++i) {
      wait_warps(3 + (i & 1), i >> 1);
      view.inv = smem_u32(INV + (i & 1) * a.inv_words + lane);
      for (int un = warp; un < units; un += EW) {  // EW <= units: at least one
        auto ready = [&]() {  // the previous tile's values are summed
          if (un == warp && i > 0) wait_warps(7, i - 1);
        };
        lanes_share<0, NC, RS, VEC, FIN>(view, un / K, un % K, mo,
                                         PART + (un % K) * a.NPR * 32 + lane, ready);
      }
      arrive(5 + (i & 1));
    }
    return;
  }
  // ---- helper warps: decode a tile ahead, sum a tile behind
  const int hw = warp - EW, dw = hw - D0, NDT = ND * 32;
  auto decode = [&](int64_t tile, int i) {  // the block's i-th tile
    const int buf = a.xbufs == 2 ? (i & 1) : 0;
    uint8_t* x = X + buf * a.xbytes;
    const int by = bytes_of(tile);
    int from = 0;
    if (bulk) {
      wait_copy(buf, (uint32_t)(a.xbufs == 2 ? i >> 1 : i) & 1);
      from = by & ~15;
    }
    // what the bulk copy leaves: a partial tile's last bytes, or, where the
    // population is not 16-byte aligned, everything
    if (from < by) {
      const uint8_t* src = a.pop + tile * (int64_t)tile_bytes;
      const int ht = tid - (EW + D0) * 32;
      if ((reinterpret_cast<uintptr_t>(src) & 15) == 0) {
        const int by16 = by & ~15;
        for (int o = from + 16 * ht; o < by16; o += 16 * NDT)
          *reinterpret_cast<uint4*>(x + o) = __ldg(reinterpret_cast<const uint4*>(src + o));
        from = by16;
      }
      for (int o = from + ht; o < by; o += NDT) x[o] = __ldg(src + o);
      bar_sync(3, NDT);
    }
    // lanes past the last chromosome decode that one again: what the buffer
    // holds behind it need not be pilots, and lanes_put takes a tile with any
    // byte of K or more apart byte by byte (2,918 chromosomes of 19 x 20: 21.2
    // us, 14.6 so)
    const int at = by == tile_bytes ? lane * LK : min(lane * LK, by - LK);
    lanes_decode(smem_u32(x) + at, smem_u32(INV + (i & 1) * a.inv_words + lane), L, K, dw, ND);
    arrive(3 + (i & 1));
    bar_sync(3, NDT);  // the buffer is read: refill it
    const int64_t nx = tile + a.xbufs * nb;
    if (bulk && dw == 0 && lane == 0 && nx < tiles && !late) issue(nx, buf);
  };
  auto sum = [&](int64_t tile, int i) {
    const int64_t n0 = tile * kLanesTile;
    lanes_sum(PART, K * a.NPR, SUMX, hw, lane, mo, a.fit + n0 * a.ntile + t, a.ntile,
              (int)min((int64_t)kLanesTile, a.n - n0));
    arrive(7);
  };
  int i = 0;
  int64_t tile = b;
  if (dw >= 0 && tile < tiles) decode(tile, 0);
  for (; tile < tiles; tile += nb, ++i) {
    if (i > 0) {  // tile i-1 is done: its values can be summed, its inverse is free
      wait_warps(5 + ((i - 1) & 1), (i - 1) >> 1);
      if (hw < 2) sum(tile - nb, i - 1);
    }
    if (dw >= 0 && tile + nb < tiles) decode(tile + nb, i + 1);
  }
  if (i > 0 && hw < 2) {
    wait_warps(5 + ((i - 1) & 1), (i - 1) >> 1);
    sum(tile - nb, i - 1);
  }
  if (late && dw == 0)  // copies issued and not waited for land (bounded) before the block ends
    for (int k = 0; k < a.xbufs; ++k)
      for (uint32_t ph = 0; ph < 2; ++ph) mbar_wait(mb0 + 8 * k, ph);
}

template <int NC, int VEC, bool FIN>
cudaError_t run_lanes(const LanesArgs& a, size_t smem, int num_sms, int64_t tiles,
                      cudaStream_t st) {
  auto kern = k_eval_f32_lanes<NC, VEC, FIN>;
  cudaError_t e = cudaSuccess;
  const int threads = (a.EW + a.NH) * 32;
  const int per_sm = cached_occupancy((const void*)kern, threads, smem, &e);
  if (e != cudaSuccess) return e;
  if (per_sm < 1) return cudaErrorInvalidConfiguration;
  // resident blocks spread evenly over the column tiles
  const int64_t want = std::max<int64_t>(1, (int64_t)per_sm * num_sms / a.ntile);
  const int64_t grid = std::min(tiles, want) * a.ntile;
  (void)cudaGetLastError();  // drop a stale error of an earlier call
  kern<<<(unsigned)grid, threads, smem, st>>>(a);
  count_launch();
  return cudaGetLastError();
}

// Instantiations for NC in [2, kLanesMaxNC], picked from a table.
template <int VEC, bool FIN, int... I>
cudaError_t pick_lanes(int NC, const LanesArgs& a, size_t smem, int sms, int64_t tiles,
                       cudaStream_t st, std::integer_sequence<int, I...>) {
  using Fn = cudaError_t (*)(const LanesArgs&, size_t, int, int64_t, cudaStream_t);
  static const Fn fn[] = {run_lanes<I + 2, VEC, FIN>...};
  if (NC < 2 || NC >= 2 + (int)sizeof...(I)) return cudaErrorNotSupported;
  return fn[NC - 2](a, smem, sms, tiles, st);
}
template <int VEC, bool FIN>
cudaError_t pick_lanes(int NC, const LanesArgs& a, size_t smem, int sms, int64_t tiles,
                       cudaStream_t st) {
  return pick_lanes<VEC, FIN>(NC, a, smem, sms, tiles, st,
                              std::make_integer_sequence<int, kLanesMaxNC - 1>{});
}

}  // namespace
}  // namespace pa
