// pa_eval_chunk.cu -- the lane-per-chromosome FP32 evaluation (paper Sec. 3.2,
// Eq. 3-6; layouts as in pa_eval_lanes.cuh) for column-tiled tables with more
// than sixteen pilots, where a tile's whole inverse (61 x 32: 62 KB) has no
// room beside the table's column tile (133 KB).
//
// Two launches.  k_eval_decode writes every tile's inverse to global memory
// once, in the layout the gather reads, eight cells (8 KB) after the other;
// k_eval_f32_chunk then holds one column tile per block and walks tiles of 32
// chromosomes: a warp per PPW pilots, whose sums for all the tile's columns
// stay in registers, so that a table word is read once per pilot; the inverse
// arrives eight cells at a time by bulk copies into a ring of four buffers.
// The warps only meet at those buffers and once per tile for the member sums.
// The user words of the block's own columns are set aside as they pass.  Sums,
// SINR steps and the member sum are those of the other FP32 kernels, bit for
// bit.
//
// What bounds it is the shared-memory data path, as in k_eval_f32_lanes: 61 x
// 32 takes 976 wavefronts per chromosome and column tile for the gathers (61
// of the 64 columns real) and ~100 for the rest; the kernel with a thread per
// (chromosome, pilot) took 1,427 (each column tile decoding again, its byte
// stores conflicting 4 deep, a byte load of the inverse per cell).  Decoding in
// the gather kernel, by four helper warps (two pilots per warp, 96 registers)
// or by all warps between chunks, was no faster than that kernel (3,057 and
// 2,857 us against 2,853): the decoding loads, 32 lines each, hold up the data
// path the gathers run through.  Measured (GB300, finite-M SINR): 2^17
// chromosomes of 61 x 32 in 2,348 us, 6,650 Gword/s of gathers, ~95 us of it the
// decode (2,853 us before), the data path 81 % busy with 1,092 wavefronts per
// chromosome and column tile.
#include <algorithm>

#include "pa_eval_lanes.cuh"

namespace pa {
namespace {

constexpr int kChunkCells = 8;
constexpr int kChunkBufs = 4;
constexpr int kChunkThreads = 1024;
constexpr int kDecodeThreads = 256;
// chromosomes whose inverses are held at once, and their bytes, at most
constexpr int64_t kChunkSlab = 1 << 17;
constexpr int64_t kChunkBytes = 256 << 20;

// Words of one chunk of one tile's inverse, and chunks per tile.
__host__ __device__ constexpr int chunk_words(int K) { return kChunkCells / 4 * K * kLanesTile; }
__host__ __device__ constexpr int chunk_count(int L) { return (L + kChunkCells - 1) / kChunkCells; }

// A piece of a chunk: sixteen users of one row of lane c's chromosome.
struct ChunkPiece {
  uint32_t v[4];
};

// Users k0 .. k0+15 of row l (x: lane c's L*K bytes in global memory); width:
// bytes per load that the rows' alignment allows (16, 4 or 1).
__device__ __forceinline__ ChunkPiece chunk_load(const uint8_t* x, int K, int l, int k0,
                                                 int width) {
  ChunkPiece p;
  const uint8_t* r = x + l * K + k0;
  if (width == 16) {  // (K is a multiple of 16)
    const uint4 q = *reinterpret_cast<const uint4*>(r);
    p.v[0] = q.x;
    p.v[1] = q.y;
    p.v[2] = q.z;
    p.v[3] = q.w;
  } else if (width == 4) {  // (K is a multiple of 4)
#pragma unroll
    for (int w = 0; w < 4; ++w)
      p.v[w] = k0 + 4 * w < K ? reinterpret_cast<const uint32_t*>(r)[w] : 0u;
  } else {
#pragma unroll
    for (int w = 0; w < 4; ++w) {
      p.v[w] = 0;
#pragma unroll
      for (int b = 0; b < 4; ++b)
        if (k0 + 4 * w + b < K) p.v[w] |= (uint32_t)r[4 * w + b] << (8 * b);
    }
  }
  return p;
}

// The piece into the inverse: byte (l & 3) of word INV[((l >> 2)*K + p)*32 + c] =
// user, dst: shared address of lane c's byte for pilot 0.  Pilots >= K are
// skipped.
__device__ __forceinline__ void chunk_put(const ChunkPiece& p, uint32_t dst, int k0, int K) {
#pragma unroll
  for (int w = 0; w < 4; ++w)
#pragma unroll
    for (int b = 0; b < 4; ++b) {
      const int k = k0 + 4 * w + b;
      const uint32_t q = (p.v[w] >> (8 * b)) & 0xffu;
      if (k < K && q < (uint32_t)K) sts8(dst + q * 128, (uint32_t)k);
    }
}

// Inverses of the chromosomes of pop (n of them): one block per (tile, chunk of
// cells), out[(tile * chunks + chunk) * chunk_words(K)].  Bytes that no row
// fills name user 0.  Bound by its reads (32 rows a chromosome apart per load)
// and its byte stores; one pass instead of one per column tile.
__global__ void __launch_bounds__(kDecodeThreads) k_eval_decode(const uint8_t* pop, int64_t n, int L,
                                                                int K, int width, uint32_t* out) {
  extern __shared__ __align__(16) uint32_t inv[];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarps = kDecodeThreads / 32;
  const int words = chunk_words(K), nch = chunk_count(L), kg = (K + 15) >> 4;
  const int64_t tile = blockIdx.x / nch;
  const int ch = (int)(blockIdx.x - tile * nch);
  for (int i = threadIdx.x; i < words / 4; i += kDecodeThreads)
    reinterpret_cast<uint4*>(inv)[i] = make_uint4(0, 0, 0, 0);
  const uint8_t* x = pop + min(tile * kLanesTile + lane, n - 1) * (L * K);
  constexpr int kU = 2;  // pieces on their way at once
  __syncthreads();
  dependents_wait();
  dependents_launch();
  for (int pc0 = warp; pc0 < kChunkCells * kg; pc0 += kU * nwarps) {
    ChunkPiece p[kU];
#pragma unroll
    for (int u = 0; u < kU; ++u) {
      const int pc = pc0 + u * nwarps, r = pc / kg, l = ch * kChunkCells + r;
      if (pc < kChunkCells * kg && l < L) p[u] = chunk_load(x, K, l, 16 * (pc - r * kg), width);
    }
#pragma unroll
    for (int u = 0; u < kU; ++u) {
      const int pc = pc0 + u * nwarps, r = pc / kg, l = ch * kChunkCells + r;
      if (pc < kChunkCells * kg && l < L)
        chunk_put(p[u], smem_u32(inv + (r >> 2) * K * 32 + lane) + (r & 3), 16 * (pc - r * kg), K);
    }
  }
  __syncthreads();
  uint4* o = reinterpret_cast<uint4*>(out + blockIdx.x * (int64_t)words);
  for (int i = threadIdx.x; i < words / 4; i += kDecodeThreads)
    o[i] = reinterpret_cast<const uint4*>(inv)[i];
}

// JT: columns of a tile; PPW: pilots per warp.  a.n chromosomes, whose inverses
// are at invg; a.fit: partial[n][ntile].  With tickets (one per tile of
// chromosomes, all zero between launches) the block that finishes a tile last
// adds its column tiles' partials in tile order into fit.
template <int JT, int PPW, bool FIN>
__global__ void __launch_bounds__(kChunkThreads, 1)
    k_eval_f32_chunk(const LanesArgs a, const uint32_t* invg, float* fit,
                     int* tickets) {
  extern __shared__ __align__(128) unsigned char smem[];
  // [0] the table's bulk copies; from 1: a buffer's chunk has landed; from
  // 1 + kChunkBufs: all warps have gathered it
  __shared__ __align__(8) uint64_t mbar[1 + 2 * kChunkBufs];
  constexpr int RS = JT + 1, NP = JT / 2, NU = JT / 4, CQ = kChunkCells / 4;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nthr = blockDim.x;
  const int L = a.L, K = a.K, LK = L * K, EW = a.EW;
  float* T = reinterpret_cast<float*>(smem);
  float* OWN = reinterpret_cast<float*>(smem + a.o_own);
  float* BN = reinterpret_cast<float*>(smem + a.o_bn);
  float* PART = reinterpret_cast<float*>(smem + a.o_part);
  float* SUMV = reinterpret_cast<float*>(smem + a.o_sum);  // [2][32][32]
  uint32_t* INV = reinterpret_cast<uint32_t*>(smem + a.o_inv);
  const int t = blockIdx.x % a.ntile;
  const int64_t b = blockIdx.x / a.ntile, nb = gridDim.x / a.ntile;
  const int jb = t * JT, jn = min(L - jb, JT);
  const int64_t tiles = (a.n + kLanesTile - 1) / kLanesTile;
  const int nch = chunk_count(L), words = a.inv_words;
  const bool mo = a.obj != 0;
  const uint32_t mb0 = smem_u32(&mbar[0]);
  const int64_t chunks = (tiles - b + nb - 1) / nb * nch;  // of this block
  // one thread: the block's q-th chunk into its buffer
  int64_t itile = b;  // of the next chunk to issue
  int ich = 0;
  auto issue = [&](int64_t q) {
    const int buf = (int)(q % kChunkBufs);
    const uint32_t mb = mb0 + 8 * (1 + buf);
    mbar_expect_tx(mb, 4 * words);
    if (!a.stall)
      bulk_g2s(smem_u32(INV + buf * words), invg + (itile * nch + ich) * words, 4 * words, mb);
    if (++ich == nch) {
      ich = 0;
      itile += nb;
    }
  };
  if (tid == 0) {
    mbar_init(mb0, 1);
    for (int i = 0; i < kChunkBufs; ++i) {
      mbar_init(mb0 + 8 * (1 + i), 1);
      mbar_init(mb0 + 8 * (1 + kChunkBufs + i), EW);
    }
    const char* src = reinterpret_cast<const char*>(a.tab + t * a.tab_floats);
    const uint32_t bytes = (uint32_t)(a.tab_floats * 4);
    mbar_expect_tx(mb0, bytes);
    constexpr uint32_t kPart = 32768;
    for (uint32_t off = 0; off < bytes; off += kPart)
      bulk_g2s(smem_u32(T) + off, src + off, min(kPart, bytes - off), mb0);
  }
  for (int i = tid; i < LK; i += nthr) OWN[i] = __ldg(a.own + i);
  for (int i = tid; i < ((L + 15) & ~15); i += nthr) BN[i] = FIN && i < L ? __ldg(a.bn + i) : 0.f;
  __syncthreads();
  // the table, which no kernel before this one in the call writes, is on its way
  // while the inverses are still decoded
  dependents_wait();
  dependents_launch();
  if (tid == 0) {
    asm volatile("fence.proxy.async;" ::: "memory");  // inverses: stores, then bulk copies
    for (int q = 0; q < kChunkBufs - 1 && q < chunks; ++q) issue(q);
  }

  // A copy that has not landed after about a second sets the error flag; the
  // warp then waits for no more of them and the block runs to the end with
  // zeros for the chunk's users (results unspecified).
  bool late = false;
  auto wait = [&](int m, uint32_t ph, int tries) {
    for (int k = 0; k < tries && !late; ++k)
      if (mbar_wait(mb0 + 8 * m, ph & 1)) return;
    if (lane == 0 && !late) atomicExch(a.err_flag, 1);
    late = true;
  };
  wait(0, 0, 2);

  const int p0 = warp * PPW;  // the last warp's pilots past K repeat K-1, unwritten
  const uint32_t T0 = smem_u32(T), KRS = 4u * K * RS;
  const f32x2 M2 = pk(a.M, a.M), pc2 = pk(a.pc, a.pc);
  // [EW*PPW][NU] words of lane c: its users in the cells of the block's own columns
  uint32_t* UW = reinterpret_cast<uint32_t*>(smem + a.o_x) + lane;
  // the tree's top: member values of a tile from its 32 partial sums
  auto close = [&](int64_t tile, int par) {
    float v[32];
#pragma unroll
    for (int k = 0; k < 32; ++k) v[k] = SUMV[(par * 32 + k) * 32 + lane];
#pragma unroll
    for (int w = 16; w > 0; w >>= 1)
#pragma unroll
      for (int k = 0; k < w; ++k) v[k] = pair_add(v[k], v[k + w], mo);
    const int64_t n = tile * kLanesTile + lane;
    if (n < a.n) a.fit[n * a.ntile + t] = v[0];
    if (!tickets) return;
    __threadfence();  // the partials before the ticket
    __syncwarp();
    int done = 0;
    if (lane == 0) done = atomicAdd(tickets + tile, 1) + 1;
    done = __shfl_sync(0xffffffffu, done, 0);
    if (done < a.ntile) return;
    __threadfence();  // the tickets before the others' partials
    if (n < a.n) {
      float s = mo ? __int_as_float(0x7f800000) : 0.f;
      for (int k = 0; k < a.ntile; ++k) {
        const float x = *reinterpret_cast<const volatile float*>(a.fit + n * a.ntile + k);
        s = mo ? fminf(s, x) : s + x;
      }
      fit[n] = s;
    }
    if (lane == 0) tickets[tile] = 0;
  };
  int64_t q = 0;  // chunks gathered
  int i = 0;      // tiles done
  for (int64_t tile = b; tile < tiles; tile += nb, ++i) {
    f32x2 acc2[PPW][NP];
    f32x2 acc1[PPW][FIN ? NP : 1];
#pragma unroll
    for (int r = 0; r < PPW; ++r)
#pragma unroll
      for (int c = 0; c < NP; ++c) {
        acc2[r][c] = 0;
        if (FIN) acc1[r][c] = 0;
      }
    uint32_t Tl = T0;
    for (int ch = 0; ch < nch; ++ch, ++q) {
      const int buf = (int)(q % kChunkBufs);
      if (warp == 0 && q + kChunkBufs - 1 < chunks) {  // refill the buffer of chunk q - 1
        if (q > 0) {
          const int64_t z = q - 1;
          wait(1 + kChunkBufs + (int)(z % kChunkBufs), (uint32_t)(z / kChunkBufs), 8);
        }
        if (lane == 0 && !late) issue(q + kChunkBufs - 1);
        __syncwarp();
      }
      wait(1 + buf, (uint32_t)(q / kChunkBufs), 2);
      const uint32_t* iv = INV + buf * words + lane;
      for (int gq = 0; gq < CQ; ++gq) {
        const int g = ch * CQ + gq, left = L - 4 * g;
        if (left <= 0) break;
        uint32_t w[PPW];
#pragma unroll
        for (int r = 0; r < PPW; ++r)
          w[r] = late ? 0u : iv[(gq * K + min(p0 + r, K - 1)) * 32];
        const int u = g - (jb >> 2);  // a quad of the block's own columns: kept
        if ((unsigned)u < (unsigned)NU)
#pragma unroll
          for (int r = 0; r < PPW; ++r) UW[((p0 + r) * NU + u) * 32] = w[r];
        auto cell = [&](int s) {
#pragma unroll
          for (int r = 0; r < PPW; ++r) {
            const uint32_t row = __dp4a(w[r], (uint32_t)(4 * RS) << (8 * s), Tl);
#pragma unroll
            for (int c = 0; c < NP; ++c) {
              const f32x2 x = pk(lds_f(row + 8 * c), lds_f(row + 8 * c + 4));
              acc2[r][c] = fma2(x, x, acc2[r][c]);
              if (FIN) acc1[r][c] = add2(acc1[r][c], x);
            }
          }
          Tl += KRS;
        };
        if (left >= 4) {
#pragma unroll
          for (int s = 0; s < 4; ++s) cell(s);
        } else {
          cell(0);
          if (left > 1) cell(1);
          if (left > 2) cell(2);
        }
      }
      __syncwarp();
      if (lane == 0) mbar_arrive(mb0 + 8 * (1 + kChunkBufs + buf));
    }
    auto finish = [&](auto mobj) {
      constexpr bool mo = decltype(mobj)::value;
#pragma unroll
      for (int r = 0; r < PPW; ++r) {
        if (p0 + r >= K) break;
        uint32_t own = smem_u32(OWN) + 4u * jb * K;
        float* part = PART + (p0 + r) * NP * 32 + lane;
        uint32_t u = 0;
#pragma unroll
        for (int c = 0; c < NP; ++c) {
          float ps = pair_init(mo);
          if (2 * c < jn) {
            if ((c & 1) == 0) u = UW[((p0 + r) * NU + (c >> 1)) * 32];
            const f32x2 bb = pk(lds_f(__dp4a(u, 4u, own)), lds_f(__dp4a(u, 4u << 8, own + 4 * K)));
            const float2 x = se_pair_f32<FIN, mo>(
                acc2[r][c], FIN ? acc1[r][c] : 0, bb,
                FIN ? lds_x2(smem_u32(BN) + 4 * jb + 8 * c) : 0, M2, pc2);
            ps = x.x;
            if (2 * c + 1 < jn) ps = pair_add(ps, x.y, mo);
          }
          own += 8 * K;
          u >>= 16;
          part[c * 32] = ps;
        }
      }
    };
    if (mo)
      finish(std::true_type{});
    else
      finish(std::false_type{});
    __syncthreads();
    if (i > 0 && warp == EW - 1) close(tile - nb, (i - 1) & 1);
    // lane v of the member sum's tree adds entries v, v + 32, ...
    for (int v = warp; v < 32; v += EW) {
      float s = pair_init(mo);
      for (int e = v; e < K * NP; e += 32) s = pair_add(s, PART[e * 32 + lane], mo);
      SUMV[((i & 1) * 32 + v) * 32 + lane] = s;
    }
    // the values are written again a tile later: behind the ring of buffers
    // when a tile has more chunks than it holds
    if (nch <= kChunkBufs) __syncthreads();
  }
  __syncthreads();
  if (i > 0 && warp == EW - 1) close(b + (i - 1) * nb, (i - 1) & 1);
  if (late && warp == 0)  // copies in flight land (bounded) before the block ends
    for (int m = 0; m <= kChunkBufs; ++m)
      for (uint32_t ph = 0; ph < 2; ++ph) mbar_wait(mb0 + 8 * m, ph);
}

template <int JT, int PPW>
cudaError_t run_chunk(const LanesArgs& a, const F32Tables& t, float* fit, int* tickets, bool fin,
                      size_t smem, int num_sms, cudaStream_t st) {
  const void* fn = fin ? (const void*)k_eval_f32_chunk<JT, PPW, true>
                       : (const void*)k_eval_f32_chunk<JT, PPW, false>;
  cudaError_t e = cudaSuccess;
  const int threads = a.EW * 32;
  const int per_sm = cached_occupancy(fn, threads, smem, &e);
  if (e != cudaSuccess) return e;
  if (per_sm < 1) return cudaErrorInvalidConfiguration;
  const int64_t tiles = (a.n + kLanesTile - 1) / kLanesTile;
  const int64_t want = std::max<int64_t>(1, (int64_t)per_sm * num_sms / a.ntile);
  const unsigned grid = (unsigned)(std::min(tiles, want) * a.ntile);
  (void)cudaGetLastError();  // drop a stale error of an earlier call
  e = launch_early(fin ? k_eval_f32_chunk<JT, PPW, true> : k_eval_f32_chunk<JT, PPW, false>, grid,
                   (unsigned)threads, smem, st, a, t.inv, fit, tickets);
  count_launch();
  return e;
}

}  // namespace

// Column-tiled tables with K > 16 (scalar rows): the fitness of n chromosomes;
// t.partial holds n * ntile values.  cudaErrorNotSupported for other tables,
// small calls (tiles_pay), or where it does not fit (shared memory, or
// device memory for the inverses of a slab of chromosomes: the context keeps
// them, at most kChunkBytes).  *summed: fit is written, else the caller adds
// the partials.  Where a block has few tiles, tickets save the launch that adds
// the partials (4 us of a generation's 78 at n = 2048, all launches ordinary); with many, the fence
// behind each tile costs more (2^17: 2,428 us against 2,348).
cudaError_t launch_eval_chunk(pa_ctx* ctx, const uint8_t* pop, int64_t n, float* fit,
                              bool* summed, cudaStream_t st) {
  F32Tables& t = ctx->t32;
  const int L = ctx->cfg.L, K = ctx->cfg.K, LK = L * K;
  const int PPW = K <= kChunkThreads / 32 ? 1 : 2;
  if (!t.streamed || t.vec != 1 || !tiles_pay(ctx, n)) return cudaErrorNotSupported;
  if (t.JT == 16 && PPW != 1) return cudaErrorNotSupported;  // (too many sums per thread)
  LanesArgs a{};
  a.ntile = t.ntile;
  a.JT = t.JT;
  a.tab_floats = t.tile_floats;
  a.NPR = t.JT / 2;
  a.EW = (K + PPW - 1) / PPW;
  a.inv_words = chunk_words(K);
  size_t b = 4 * (size_t)a.tab_floats;
  a.o_own = (int)b;
  b += 4 * (size_t)((LK + 3) & ~3);
  a.o_bn = (int)b;
  b += 4 * (size_t)((L + 15) & ~15);
  a.o_part = (int)b;
  b += 4 * (size_t)K * a.NPR * kLanesTile;
  a.o_sum = (int)b;
  b += 2 * 4 * 32 * kLanesTile;
  a.o_inv = (int)b;
  b += kChunkBufs * 4 * (size_t)a.inv_words;
  a.o_x = (int)b;
  b += 4 * (size_t)a.EW * PPW * (t.JT / 4) * kLanesTile;
  if (b + 1024 > (size_t)kSmemBudget) return cudaErrorNotSupported;
  const int nch = chunk_count(L);
  const int64_t tile_bytes = 4 * (int64_t)a.inv_words * nch;
  const int64_t slab = std::min({n, kChunkSlab, kChunkBytes / tile_bytes * kLanesTile});
  const int64_t slab_tiles = (slab + kLanesTile - 1) / kLanesTile;
  if (t.inv_cap < slab_tiles) {
    // not while the stream is captured (an allocation would end the capture), nor
    // again where it failed
    cudaStreamCaptureStatus cap = cudaStreamCaptureStatusActive;
    if (cudaStreamIsCapturing(st, &cap) != cudaSuccess) (void)cudaGetLastError();
    if (cap != cudaStreamCaptureStatusNone || t.inv_none <= slab_tiles)
      return cudaErrorNotSupported;
    cudaFree(t.inv);
    t.inv = nullptr;
    t.inv_cap = 0;
    const size_t inv_bytes = (size_t)(tile_bytes * slab_tiles);
    if (cudaMalloc(&t.inv, inv_bytes + sizeof(int) * slab_tiles) != cudaSuccess) {
      (void)cudaGetLastError();
      t.inv_none = slab_tiles;
      return cudaErrorNotSupported;
    }
    t.tickets = reinterpret_cast<int*>(reinterpret_cast<unsigned char*>(t.inv) + inv_bytes);
    const cudaError_t e = cudaMemsetAsync(t.tickets, 0, sizeof(int) * slab_tiles, st);
    if (e != cudaSuccess) return e;
    t.inv_cap = slab_tiles;
  }
  a.tab = t.tab;
  a.own = t.own;
  a.bn = t.bn;
  a.err_flag = t.err_flag;
  a.L = L;
  a.K = K;
  a.M = t.M;
  a.pc = t.pc;
  a.obj = ctx->cfg.objective;
  const bool fin = ctx->cfg.mode == PA_SINR_FINITE_M;
  *summed = n <= slab && slab_tiles * t.ntile <= 4 * (int64_t)ctx->num_sms;
  int* tickets = *summed ? t.tickets : nullptr;
  for (int64_t n0 = 0; n0 < n; n0 += slab) {
    a.n = std::min(slab, n - n0);
    a.fit = t.partial + n0 * t.ntile;
    a.stall = ctx->test_stall;
    ctx->test_stall = 0;
    const uint8_t* x = pop + n0 * LK;
    const uintptr_t base = reinterpret_cast<uintptr_t>(x);
    const int width = K % 16 == 0 && base % 16 == 0 ? 16 : K % 4 == 0 && base % 4 == 0 ? 4 : 1;
    const int64_t tiles = (a.n + kLanesTile - 1) / kLanesTile;
    (void)cudaGetLastError();  // drop a stale error of an earlier call
    cudaError_t e = launch_early(k_eval_decode, (unsigned)(tiles * nch), kDecodeThreads,
                                 4 * (size_t)a.inv_words, st, x, a.n, L, K, width, t.inv);
    count_launch();
    if (e != cudaSuccess) return e;
    switch (t.JT * 10 + PPW) {
      case 161: e = run_chunk<16, 1>(a, t, fit + n0, tickets, fin, b, ctx->num_sms, st); break;
      case 81: e = run_chunk<8, 1>(a, t, fit + n0, tickets, fin, b, ctx->num_sms, st); break;
      case 82: e = run_chunk<8, 2>(a, t, fit + n0, tickets, fin, b, ctx->num_sms, st); break;
      case 41: e = run_chunk<4, 1>(a, t, fit + n0, tickets, fin, b, ctx->num_sms, st); break;
      case 42: e = run_chunk<4, 2>(a, t, fit + n0, tickets, fin, b, ctx->num_sms, st); break;
      default: return cudaErrorInvalidValue;
    }
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

}  // namespace pa
