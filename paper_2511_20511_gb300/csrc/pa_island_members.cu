// pa_island_members.cu -- population K-means of the island GA (Alg. 2's
// re-clustering) on a cluster with the members split over the CTAs: the form for
// many members of few users.
//
// CTA r of R assigns members [N r / R, N (r+1) / R); every CTA holds the whole
// staged population and its own copy of the counts, Q, m and the initial
// centroids (all computed identically).  A pass: assignment of the own slice, the
// changed members listed per CTA; one cluster barrier; every CTA reads the other
// CTAs' changed lists and cluster sizes (distributed shared memory), decides the
// same stop, and replays all changed members into its counts.  Lists and sizes are
// double-buffered by pass parity, so a CTA can list the next pass's changes while
// another still reads this pass's.
//
// The form with the users split (pa_island_kmeans.cuh) pushes every member's sums
// from every CTA and works in few words of users here: per pass, that form /
// this one, 7 x 4 at N = 1000, C = 9: 14.5 / 8.9 us; N = 4000, C = 17: 277 / 14; 7 x
// 10 at N = 2000, C = 17: 31.9 / 22.2; but 7 x 10 at N = 1000, C = 9: 11.4 / 14.4, 19 x
// 10 at N = 256, C = 5: 5.3 / 11.4.
#include <algorithm>

#include "pa_island_kmeans.cuh"

namespace pa {
namespace {

constexpr int kMbThreads = 1024;
constexpr int kMbClusterMax = 8;  // portable cluster sizes

struct MbLayout {
  int NP, W, us, Nr;
  size_t o_lab, o_chg, o_gchg, o_cnt, o_sb, o_pw, total;
};

MbLayout mb_layout(int N, int L, int K, int C, int R, int us) {
  MbLayout k;
  const size_t LK = (size_t)L * K;
  const int CWp = ((C + 1) / 2) | 1;
  const size_t N4 = (size_t)((N + 3) & ~3);
  k.NP = N | 1;
  k.W = (int)((LK + 3) / 4);
  k.us = us;
  k.Nr = (N + R - 1) / R;
  size_t b = 0;
  k.o_lab = b;   // [N] labels of the own slice (whole range allocated)
  b += 4 * N4;   // + [N] initial permutation
  b += 4 * N4;
  k.o_chg = b;   // [2][N] own changed members per pass parity
  b += 4 * 2 * N4;
  k.o_gchg = b;  // [N] every CTA's changed members of this pass
  b += 4 * N4;
  k.o_cnt = b;
  b += 4 * LK * K * CWp;
  k.o_sb = b;
  if (us > 1) b += 4 * (size_t)us * C * k.Nr;
  b = (b + 15) & ~size_t(15);
  k.o_pw = b;
  b += 4 * (size_t)k.W * k.NP;
  k.total = (b + 15) & ~size_t(15);
  return k;
}

// Per-CTA scalars of a cluster K-means (shared memory).
struct MbShared {
  unsigned long long Q[kMaxIslands];   // sum of squared counts per cluster
  int m[kMaxIslands];                  // centroid sizes
  int nm[kMaxIslands];                 // sizes of the new partition (all CTAs)
  int live[kMaxIslands];               // the cluster has members in the new partition
  int stale[kMaxIslands];              // its counts are not the sum over its members
  uint32_t rdraw[kMaxIslands];         // initial-centroid draws
  int nm_own[2][kMaxIslands];          // own slice's sizes, per pass parity
  int nchg_own[2];                     // own slice's changed members, per pass parity
  int cnt_r[kMbClusterMax];            // changed members of each CTA in this pass
};

// Shared-memory arrays of a cluster K-means (MbLayout).
struct MbView {
  MbShared* sh;
  uint32_t* pw;   // [W][NP] staged pilots (clamped below K), filled by the stage
  int NP;
  uint32_t* cnt;  // [L*K*K][CWp] packed 16-bit count pairs
  int CWp;
  int* lab;       // [N] labels (the own slice's are final at return)
  int* perm;      // [N] initial permutation
  int* chg;       // [2][N4] own changed members per pass parity
  int* gchg;      // [N] every CTA's changed members of a pass
  int* sb;        // [us][C][Nr] partial sums of the user splits
  int us, Nr;
};

// One population K-means on the calling cluster (every CTA calls it, all
// threads); stage(warp, nwarps, lane) fills v.pw, run by warps 0..nwarps-1
// (= all warps but the last, which makes the initial draws meanwhile).
// Returns the number of assignment passes; the labels of CTA r's slice
// [N r / R, N (r+1) / R) are in its v.lab.  The caller keeps the CTAs
// alive (a cluster barrier) while others may still read this CTA's lists.
template <typename Stage>
__device__ __forceinline__ int km_members(const MbView& kv, const KmParams& p,
                                          cg::cluster_group& cluster, Stage stage) {
  MbShared& sh = *kv.sh;
  const int R = (int)cluster.num_blocks(), rank = (int)cluster.block_rank();
  const int N = p.N, K = p.K, C = p.C, LK = p.L * p.K, LKK = LK * p.K;
  const int CW = (C + 1) >> 1, CWp = kv.CWp, NP = kv.NP, W = (LK + 3) >> 2, us = kv.us;
  const int tid = threadIdx.x, nthr = blockDim.x, lane = tid & 31, warp = tid >> 5;
  const int nwarps = nthr >> 5;
  const unsigned full = 0xffffffffu;
  const int n_lo = N * rank / R, n_hi = N * (rank + 1) / R;  // N * R < 2^31
  const int Nr = kv.Nr;
  int* lab = kv.lab;
  int* perm = kv.perm;
  int* chg = kv.chg;
  int* gchg = kv.gchg;
  uint32_t* cnt = kv.cnt;
  int* sb = kv.sb;
  uint32_t* pw = kv.pw;
  const int N4 = (N + 3) & ~3;
  if (warp == nwarps - 1) {
    for (int c = lane; c < C; c += 32) {
      DrawStream ds(p.seed, 0, (uint64_t)p.gen, kTagIsland);
      sh.rdraw[c] = below(ds.draw((uint32_t)c), (uint32_t)(N - c));
    }
  } else {
    const int st = nthr - 32;
    stage(warp, nwarps - 1, lane);
    for (int i = tid; i < LKK * CWp; i += st) cnt[i] = 0;
    for (int n = tid; n < N; n += st) {
      perm[n] = n;
      lab[n] = -1;
    }
    if (tid < kMaxIslands) {
      sh.Q[tid] = 0ULL;
      sh.stale[tid] = 1;
      sh.nm_own[0][tid] = 0;
      sh.nm_own[1][tid] = 0;
    }
    if (tid < 2) sh.nchg_own[tid] = 0;
  }
  __syncthreads();
  if (tid == 0) {
    for (int c = 0; c < C; ++c) {
      const int j = c + (int)sh.rdraw[c];
      const int t = perm[c];
      perm[c] = perm[j];
      perm[j] = t;
      sh.m[c] = 1;
    }
  }
  __syncthreads();
  for (int c = warp; c < C; c += nwarps) {
    const int n = perm[c], h = (c & 1) * 16;
    unsigned long long dq = 0;
    for (int u = lane; u < LK; u += 32) {
      const int x = km_pilot<true>(pw, NP, nullptr, LK, K, n, u);
      const uint32_t o = atomicAdd(cnt + (u * K + x) * CWp + (c >> 1), 1u << h);
      dq += (unsigned long long)(2 * km_half(o, h) + 1);
    }
    dq = warp_sum_u64(dq);
    if (lane == 0) atomicAdd(&sh.Q[c], dq);
  }
  __syncthreads();
  const int G = (n_hi - n_lo + 31) >> 5;
  const int wblk = max(1, 65535 / (4 * N));
  auto fold = [&](int c, long long S, int& best, long long& bd) {
    const long long mc = sh.m[c];
    const long long A = (long long)LK * mc * mc - 2 * mc * S + (long long)sh.Q[c];
    const long long mb = sh.m[best];
    if (c == 0 || A * mb * mb < bd * mc * mc) {
      best = c;
      bd = A;
    }
  };
  auto record = [&](int n, int best, int par) {
    const bool valid = n < n_hi;
    const int old = valid ? lab[n] : 0;
    const bool moved = valid && old != best;
    const unsigned bm = __ballot_sync(full, moved);
    if (bm) {
      const int leader = __ffs(bm) - 1;
      int base = 0;
      if (lane == leader) base = atomicAdd(&sh.nchg_own[par], __popc(bm));
      base = __shfl_sync(full, base, leader);
      if (moved)
        chg[par * N4 + base + __popc(bm & ((1u << lane) - 1u))] = (n << 13) | ((old + 1) << 6) | best;
    }
    const unsigned same = __match_any_sync(full, valid ? best : -1 - lane);
    if (valid) {
      lab[n] = best;
      if ((int)(__ffs(same) - 1) == lane) atomicAdd(&sh.nm_own[par][best], __popc(same));
    }
  };
  int passes = 0;
  for (int it = 0; it < p.max_iter; ++it) {
    const int par = it & 1;
    // ---- assignment of the own slice
    for (int t = warp; t < G * us; t += nwarps) {
      const int g = t / us, s = t - g * us;
      const int n = n_lo + g * 32 + lane;
      const int nn = n < n_hi ? n : n_hi - 1;
      const int w0 = W * s / us, w1 = W * (s + 1) / us;
      int best = 0;
      long long bd = 0;
      for (int c0 = 0; c0 < C; c0 += 2 * kKmMaxW) {
        int S[2 * kKmMaxW];
        const int i0 = c0 >> 1;
        switch (min(kKmMaxW, CW - i0)) {
#define PA_KM_CASE(NW)                                                                    \
  case NW:                                                                                \
    km_sums<NW, true>(S, cnt, CWp, i0, K, LK, w0, w1, wblk, pw, NP, nullptr, nn);           \
    break;
          PA_KM_CASE(1)
          PA_KM_CASE(2)
          PA_KM_CASE(3)
          PA_KM_CASE(4)
          PA_KM_CASE(5)
          PA_KM_CASE(6)
          PA_KM_CASE(7)
          default:
            km_sums<8, true>(S, cnt, CWp, i0, K, LK, w0, w1, wblk, pw, NP, nullptr, nn);
#undef PA_KM_CASE
        }
#pragma unroll
        for (int q = 0; q < 2 * kKmMaxW; ++q) {
          const int c = c0 + q;
          if (c < C) {
            if (us > 1) {
              if (n < n_hi) sb[(s * C + c) * Nr + (n - n_lo)] = S[q];
            } else {
              fold(c, S[q], best, bd);
            }
          }
        }
      }
      if (us == 1) record(n, best, par);
    }
    __syncthreads();
    if (us > 1) {
      for (int n0 = n_lo + warp * 32; n0 < n_hi; n0 += nthr) {
        const int n = n0 + lane;
        int best = 0;
        long long bd = 0;
        if (n < n_hi)
          for (int c = 0; c < C; ++c) {
            int S = 0;
            for (int s = 0; s < us; ++s) S += sb[(s * C + c) * Nr + (n - n_lo)];
            fold(c, S, best, bd);
          }
        record(n, best, par);
      }
    }
    // ---- every CTA's labels, lists and sizes of this pass are visible
    cluster.sync();
    if (tid < R) sh.cnt_r[tid] = *cluster.map_shared_rank(&sh.nchg_own[par], tid);
    if (tid >= 32 && tid < 32 + C) {
      const int c = tid - 32;
      int v = 0;
      for (int r = 0; r < R; ++r) v += *cluster.map_shared_rank(&sh.nm_own[par][c], r);
      sh.nm[c] = v;
    }
    __syncthreads();
    int total = 0;
    for (int r = 0; r < R; ++r) total += sh.cnt_r[r];
    ++passes;
    if (total == 0 || it == p.max_iter - 1) break;
    // every CTA's changed members, in CTA order
    for (int k = tid; k < total; k += nthr) {
      int r = 0, base = 0;
      while (k >= base + sh.cnt_r[r]) {
        base += sh.cnt_r[r];
        ++r;
      }
      gchg[k] = *cluster.map_shared_rank(chg + par * N4 + (k - base), r);
    }
    for (int e = tid; e < LKK; e += nthr)
      for (int i = 0; i < CW; ++i) {
        const bool z0 = sh.stale[2 * i] && sh.nm[2 * i] > 0;
        const bool z1 = 2 * i + 1 < C && sh.stale[2 * i + 1] && sh.nm[2 * i + 1] > 0;
        if (z0 || z1) cnt[e * CWp + i] &= (z0 ? 0u : 0xffffu) | (z1 ? 0u : 0xffff0000u);
      }
    if (tid < C) {
      sh.live[tid] = sh.nm[tid] > 0;
      if (sh.nm[tid] > 0) {
        if (sh.stale[tid]) sh.Q[tid] = 0ULL;
        sh.m[tid] = sh.nm[tid];
      }
    }
    // the other parity's own lists were last read before this pass's barrier
    if (tid < kMaxIslands) sh.nm_own[par ^ 1][tid] = 0;
    if (tid == 0) sh.nchg_own[par ^ 1] = 0;
    __syncthreads();
    for (int k = warp; k < total; k += nwarps) {
      const int e = gchg[k], n = e >> 13, A = ((e >> 6) & 127) - 1, Bc = e & 63;
      const bool sub = A >= 0 && sh.live[A];
      const int hb = (Bc & 1) * 16, ha = (A & 1) * 16;
      uint32_t* pb = cnt + (Bc >> 1);
      uint32_t* pold = cnt + (sub ? A >> 1 : 0);
      unsigned long long dqb = 0, dqa = 0;
      for (int u = lane; u < LK; u += 32) {
        const int o = (u * K + km_pilot<true>(pw, NP, nullptr, LK, K, n, u)) * CWp;
        const uint32_t ob = atomicAdd(pb + o, 1u << hb);
        dqb += (unsigned long long)(2 * km_half(ob, hb) + 1);
        if (sub) {
          const uint32_t oa = atomicAdd(pold + o, 0u - (1u << ha));
          dqa += (unsigned long long)(1 - 2 * km_half(oa, ha));
        }
      }
      dqb = warp_sum_u64(dqb);
      dqa = warp_sum_u64(dqa);
      if (lane == 0) {
        atomicAdd(&sh.Q[Bc], dqb);
        if (sub) atomicAdd(&sh.Q[A], dqa);
      }
    }
    if (tid < C) sh.stale[tid] = sh.nm[tid] == 0;
    __syncthreads();
  }
  return passes;
}

struct MbArgs {
  const uint8_t* pop;  // [N][LK]
  KmParams p;
  MbLayout k;
  int32_t* label;      // [N] out
  int32_t* passes;     // [1] out
};

__global__ void __launch_bounds__(kMbThreads) k_island_kmeans_mb(const MbArgs a) {
  cg::cluster_group cluster = cg::this_cluster();
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ MbShared sh;
  const int N = a.p.N, K = a.p.K, LK = a.p.L * K, W = a.k.W, NP = a.k.NP;
  MbView v;
  v.sh = &sh;
  v.pw = reinterpret_cast<uint32_t*>(smem + a.k.o_pw);
  v.NP = NP;
  v.cnt = reinterpret_cast<uint32_t*>(smem + a.k.o_cnt);
  v.CWp = km_cwp(a.p.C);
  v.lab = reinterpret_cast<int*>(smem + a.k.o_lab);
  v.perm = v.lab + ((N + 3) & ~3);
  v.chg = reinterpret_cast<int*>(smem + a.k.o_chg);
  v.gchg = reinterpret_cast<int*>(smem + a.k.o_gchg);
  v.sb = reinterpret_cast<int*>(smem + a.k.o_sb);
  v.us = a.k.us;
  v.Nr = a.k.Nr;
  uint32_t* pw = v.pw;
  const uint8_t* pop = a.pop;
  // word w of member n holds the pilots of users 4w .. 4w+3
  const int passes = km_members(v, a.p, cluster, [&](int warp, int sw, int lane) {
    for (int n = warp; n < N; n += sw) {
      const uint8_t* X = pop + (int64_t)n * LK;
      for (int w = lane; w < W; w += 32) {
        uint32_t x = 0;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          const int u = 4 * w + j;
          x |= (uint32_t)(u < LK ? min((int)X[u], K - 1) : K - 1) << (8 * j);
        }
        pw[w * NP + n] = x;
      }
    }
  });
  const int R = (int)cluster.num_blocks(), rank = (int)cluster.block_rank();
  const int n_lo = N * rank / R, n_hi = N * (rank + 1) / R;  // N * R < 2^31
  for (int n = n_lo + (int)threadIdx.x; n < n_hi; n += blockDim.x) a.label[n] = v.lab[n];
  if (rank == 0 && threadIdx.x == 0 && a.passes) *a.passes = passes;
  cluster.sync();  // the other CTAs may still read this CTA's lists
}

}  // namespace

// R = min(8, N/32) CTAs, each holding the whole population and its own counts.
// cudaErrorNotSupported when it does not pay (above) or apply (fewer than 64
// members, a layout beyond shared memory, a cluster shape that cannot be
// resident).  The lines, in members per word of four users, lie between the
// measured changes of side (us per pass, this form / the other): up to 8 clusters
// 7 x 4 at 57 (8.8 / 7.6) and 143 (7.8 / 11.0), 7 x 10 at 111 (13.3 / 11.0), and under
// four words the other form's whatever N (2 x 2, N = 4000: 67 / 67); 9 to 16, 7 x 4 at
// 57 (9.0 / 9.0), 7 x 10 at 56 (14.4 / 11.4) and 111 (13.9 / 16.6); 17 to 32, 7 x 4 at 57
// (12.6 / 15.2), 7 x 10 at 56 (21.1 / 19.2); above, 7 x 4 at 57 (35.2 / 28.6) and 143 (33.1
// / 46.6).
cudaError_t launch_island_kmeans_mb(const pa_ctx* ctx, const uint8_t* pop, int gen, int32_t* labels,
                                    cudaStream_t st) {
  const pa_config& c = ctx->cfg;
  const int W = (c.L * c.K + 3) / 4;
  const int line = c.islands <= 8 ? 120 : c.islands > 16 && c.islands <= 32 ? 56 : 80;
  if (c.N < 64 || (c.islands <= 8 && W < 4) || c.N <= line * W) return cudaErrorNotSupported;
  const int R = std::min(kMbClusterMax, std::max(2, c.N / 32));
  const int groups = ((c.N + R - 1) / R + 31) / 32;
  const size_t budget = (size_t)kSmemBudget - 4096;  // beside the static arrays
  int us = std::max(1, std::min({kKmSplits, kMbThreads / 32 / groups, W}));
  while (us > 1 && mb_layout(c.N, c.L, c.K, c.islands, R, us).total > budget) --us;
  MbArgs a;
  a.k = mb_layout(c.N, c.L, c.K, c.islands, R, us);
  if (a.k.total > budget) return cudaErrorNotSupported;
  cudaLaunchAttribute attr[1];
  cudaLaunchConfig_t cfg = cluster_config(R, kMbThreads, a.k.total, st, attr);
  bool ok = false;
  cudaError_t e = cluster_resident((const void*)k_island_kmeans_mb, ctx->device, cfg, &ok);
  if (e != cudaSuccess) return e;
  if (!ok) return cudaErrorNotSupported;
  a.pop = pop;
  a.p = KmParams{c.N, c.L, c.K, c.islands, c.island_iter, c.seed, gen};
  a.label = labels;
  a.passes = ctx->isl_passes;
  (void)cudaGetLastError();  // drop a stale error of an earlier call
  e = cudaLaunchKernelEx(&cfg, k_island_kmeans_mb, a);
  count_launch();
  return e;
}

}  // namespace pa
