// pa_island_kmeans.cuh -- device code of the population K-means of the
// island GA (Alg. 2's re-clustering): the count-based assignment helpers
// and the cluster form of the Lloyd iteration, shared by the K-means
// kernels (pa_island.cu) and the fused solve's island mode
// (pa_solve_island.cu), which stage the population differently (from
// global memory, or from the cluster's member records).
#pragma once
#include <cooperative_groups.h>

#include <algorithm>

#include "pa_internal.cuh"

namespace pa {
namespace {

namespace cg = cooperative_groups;

constexpr int kKmMaxW = 8;   // pair words of counts one lane sums at once (16 clusters)
constexpr int kKmSplits = 8; // most warps sharing one group of 32 members (user ranges)

__device__ __forceinline__ unsigned long long warp_sum_u64(unsigned long long v) {
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
  return v;
}

// Sum over a warp of values below 2^48 (two halves of 24 bits, each summed in
// one instruction).
__device__ __forceinline__ unsigned long long warp_sum_u48(unsigned long long v) {
  const uint32_t lo = __reduce_add_sync(0xffffffffu, (uint32_t)v & 0xffffffu);
  const uint32_t hi = __reduce_add_sync(0xffffffffu, (uint32_t)(v >> 24));
  return ((unsigned long long)hi << 24) + lo;
}

// Pilot of user u of member n (a pilot >= K reads as K-1): from the staged
// words (clamped when staged), or from the rows.
template <bool PS>
__device__ __forceinline__ int km_pilot(const uint32_t* pw, int NP, const uint8_t* pop, int LK,
                                        int K, int n, int u) {
  if (PS) return (int)((pw[(u >> 2) * NP + n] >> (8 * (u & 3))) & 0xffu);
  return min((int)pop[(int64_t)n * LK + u], K - 1);
}

// Word w of member n: the (clamped) pilots of users 4w .. 4w+3, low byte
// first; bytes past the row end are K-1.
template <bool PS>
__device__ __forceinline__ uint32_t km_word(const uint32_t* pw, int NP, const uint8_t* pop, int LK,
                                            int K, int n, int w) {
  if (PS) return pw[w * NP + n];
  uint32_t v = 0;
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    const int u = 4 * w + j;
    v |= (uint32_t)(u < LK ? min((int)pop[(int64_t)n * LK + u], K - 1) : K - 1) << (8 * j);
  }
  return v;
}

// S(n, c) for the 2*NW clusters of pair words i0 .. i0+NW-1 over the users
// of words w0 .. w1-1: a lane sums packed 16-bit pairs (one load serves two
// clusters) for wblk words at a time -- a half stays below 2^16 since each
// count is at most N -- and widens them into S.  Words below wfull hold
// four users each; only the row's last word is checked.
template <int NW, bool PS>
__device__ __forceinline__ void km_sums(int (&S)[2 * kKmMaxW], const uint32_t* cnt, int CWp,
                                        int i0, int K, int LK, int w0, int w1, int wblk,
                                        const uint32_t* pw, int NP, const uint8_t* pop, int n) {
  const int wfull = LK >> 2, KC = K * CWp;
#pragma unroll
  for (int q = 0; q < 2 * NW; ++q) S[q] = 0;
  for (int wb = w0; wb < w1; wb += wblk) {
    const int we = min(w1, wb + wblk);
    uint32_t P[NW];
#pragma unroll
    for (int i = 0; i < NW; ++i) P[i] = 0;
    int w = wb;
    for (; w < min(we, wfull); ++w) {
      const uint32_t v = km_word<PS>(pw, NP, pop, LK, K, n, w);
      const uint32_t* row = cnt + 4 * w * KC + i0;
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const uint32_t* e = row + j * KC + (int)((v >> (8 * j)) & 0xffu) * CWp;
#pragma unroll
        for (int i = 0; i < NW; ++i) P[i] += e[i];
      }
    }
    for (; w < we; ++w) {  // the row's last, partial word
      const uint32_t v = km_word<PS>(pw, NP, pop, LK, K, n, w);
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const int u = 4 * w + j;
        if (u < LK) {
          const uint32_t* e = cnt + u * KC + (int)((v >> (8 * j)) & 0xffu) * CWp + i0;
#pragma unroll
          for (int i = 0; i < NW; ++i) P[i] += e[i];
        }
      }
    }
#pragma unroll
    for (int i = 0; i < NW; ++i) {
      S[2 * i] += (int)(P[i] & 0xffffu);
      S[2 * i + 1] += (int)(P[i] >> 16);
    }
  }
}

// Half h (0: low, 16: high) of a packed word.
__device__ __forceinline__ long long km_half(uint32_t v, int h) {
  return (long long)((v >> h) & 0xffffu);
}

// The cluster form of the K-means (k_island_kmeans_cl, and the fused solve in
// island mode).  The users are split: CTA r of R stages the pilots of every
// member for its words of four users [W r / R, W (r+1) / R) only, and keeps
// the counts of those users.  A pass:
//   1. each CTA sums S(n, c) over its users for all members (a lane a member,
//      packed pairs of clusters) and pushes the sums, and its share of Q, to
//      the CTA that owns the member (n in [N r / R, N (r+1) / R));
//   2. cluster barrier; the owners add the R shares, take the nearest
//      centroids and push their members' labels to every CTA;
//   3. cluster barrier; every CTA finds the changed members and the sizes
//      from the labels, so all take the same decision to stop, and moves the
//      changed members' one-hots in the counts of its own users.
// What bounds a pass is latency: two cluster barriers, four block barriers
// and a chain of short phases.  Splitting the members instead (each CTA
// assigning a slice and replaying every changed member over all L*K users into
// a full copy of the counts) has one cluster barrier less, but each CTA then
// stages the whole population and repeats all updates: 64 us per re-clustering
// of 256 x 190 into 5 islands in the fused solve (5.2 passes), 54 us alone,
// against 30 and 25 us here; the island solve of 200 generations 5.49 -> 3.26
// ms (with the elites found by their slots' warps, which took 0.4 of it).
constexpr int kKmChunk = 8;  // pair words of S pushed at once (16 clusters)

// Words per (user, pilot) entry of the counts: ceil(C/2), rounded up to odd.
__host__ __device__ constexpr int km_cwp(int C) { return ((C + 1) / 2) | 1; }

// Shared-memory layout of a cluster K-means (byte offsets from a 16-byte
// aligned base) of N members on R CTAs of `threads` threads; smaller chunks of
// S when the total would exceed `budget` (the caller checks that it fits).
struct KmClLayout {
  int NP, wown, us, qs, es, CWc, nbuf;
  int o_lab, o_nlab, o_own, o_chg, o_cnt, o_pw, o_in, o_q, o_s, total;
};

inline KmClLayout km_cl_layout(int N, int L, int K, int C, int R, int threads, int budget,
                               int chunk = kKmChunk) {
  KmClLayout k;
  const int LK = L * K, W = (LK + 3) / 4, CW = (C + 1) / 2;
  const int N4 = (N + 3) & ~3;
  k.NP = N | 1;
  k.wown = (W + R - 1) / R;
  const int Nr = (N + R - 1) / R;
  // splits of a CTA's words: enough for its threads, and few enough users per
  // split that a packed 16-bit sum of counts <= N cannot overflow
  const int wmax = std::max(1, 65535 / (4 * N));
  k.us = std::max((k.wown + wmax - 1) / wmax,
                  std::min(k.wown, std::max(1, threads / ((N + 31) & ~31))));
  k.CWc = std::min(chunk, CW > 4 ? 8 : CW > 2 ? 4 : CW);
  k.nbuf = CW > k.CWc ? 2 : 1;
  // splits of the Q sums (a warp a pair of clusters and split)
  k.qs = std::max(1, std::min(threads / 32 / CW, (4 * k.wown * K + 255) / 256));
  // words from one share of the sums to the next: the owner's lanes read one
  // member's words of 32 / CWc shares at once, CWc words (a bank group) apart
  k.es = Nr * k.CWc + (32 - Nr * k.CWc % 32 + k.CWc) % 32;
  int b = 0;
  auto take = [&](int& o, int64_t bytes) {
    o = b;
    b = (int)std::min<int64_t>((b + bytes + 15) & ~int64_t(15), 1 << 29);
  };
  take(k.o_lab, 4 * N4);   // labels
  take(k.o_nlab, 4 * N4);  // a pass's new labels (pushed by the owners)
  take(k.o_own, 4 * N4);   // owner << 16 | place in its slice
  take(k.o_chg, 4 * N4);   // changed members (and the initial permutation)
  take(k.o_cnt, 16LL * k.wown * K * km_cwp(C));
  take(k.o_pw, 4LL * k.wown * k.NP);
  take(k.o_in, 4LL * k.nbuf * R * k.us * k.es);  // [nbuf][R*us][Nr][CWc] (pitch es)
  take(k.o_q, 8LL * R * k.qs * C);               // [R*qs][C] shares of Q
  take(k.o_s, 4LL * Nr * C);                     // [Nr][C] sums of the own slice
  k.total = b;
  if (b > budget && k.CWc > 1)
    return km_cl_layout(N, L, K, C, R, threads, budget, k.CWc / 2);
  return k;
}

// Per-CTA scalars of a cluster K-means (shared memory).
struct KmShared {
  unsigned long long Q[kMaxIslands];   // sums of squared counts
  int m[kMaxIslands];                  // centroid sizes
  int nm[kMaxIslands];                 // sizes of the new partition
  int stale[kMaxIslands];              // its counts are not the sum over its members
  uint32_t rdraw[kMaxIslands];         // initial-centroid draws
  int nchg;                            // changed members of the pass
};

// Shared-memory arrays of a cluster K-means (KmClLayout).
struct KmView {
  KmShared* sh;
  unsigned char* base;
  KmClLayout k;
};

struct KmParams {
  int N, L, K, C, max_iter;
  uint64_t seed;
  int gen;
};

__device__ __forceinline__ uint32_t km_mapa(const void* local, int rank) {
  uint32_t a = (uint32_t)__cvta_generic_to_shared(local), r;
  asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(rank));
  return r;
}
__device__ __forceinline__ void km_st(uint32_t addr, uint32_t v) {
  asm volatile("st.shared::cluster.u32 [%0], %1;" ::"r"(addr), "r"(v) : "memory");
}
__device__ __forceinline__ void km_st64(uint32_t addr, unsigned long long v) {
  asm volatile("st.shared::cluster.u64 [%0], %1;" ::"r"(addr), "l"(v) : "memory");
}
__device__ __forceinline__ void km_st128(uint32_t addr, uint32_t x, uint32_t y, uint32_t z,
                                         uint32_t w) {
  asm volatile("st.shared::cluster.v4.u32 [%0], {%1, %2, %3, %4};" ::"r"(addr), "r"(x), "r"(y),
               "r"(z), "r"(w)
               : "memory");
}

// Member n's packed sums over the staged words w0 .. w1-1 for the pair words
// i0 .. i0+NW-1, pushed to address `to` (CWc words there).  Users past L*K in
// the last word read pilot 0 and have counts of zero.
template <int NW>
__device__ __forceinline__ void km_push(const uint32_t* cnt, int CWp, int K, const uint32_t* pw,
                                        int NP, int n, int w0, int w1, int i0, int CWc,
                                        uint32_t to) {
  const int KC = K * CWp;
  uint32_t P[8];
#pragma unroll
  for (int i = 0; i < 8; ++i) P[i] = 0;
  for (int w = w0; w < w1; ++w) {
    const uint32_t v = pw[w * NP + n];
    const uint32_t* row = cnt + 4 * w * KC + i0;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const uint32_t* e = row + j * KC + (int)((v >> (8 * j)) & 0xffu) * CWp;
#pragma unroll
      for (int i = 0; i < NW; ++i) P[i] += e[i];
    }
  }
  if (CWc >= 4) {
    km_st128(to, P[0], P[1], P[2], P[3]);
    if (CWc > 4) km_st128(to + 16, P[4], P[5], P[6], P[7]);
  } else {
    km_st(to, P[0]);
    if (CWc > 1) km_st(to + 4, P[1]);
  }
}

// One population K-means on the calling cluster (every CTA calls it, all
// threads); stage(pw, NP, wb, nw) fills pw[w * NP + n], w < nw, with the pilots
// (clamped below K; 0 past the row) of users 4 (wb + w) .. + 3 of every member,
// run by all threads but the last warp's (which makes the initial draws
// meanwhile).  Returns the number of assignment passes; every CTA then holds
// all labels (o_lab) and the clusters' sizes (sh.nm).  The CTAs' shared
// memory may be read and written by the others until the last cluster
// barrier of the call only.
// started(): called by all threads before the first access to another CTA's
// shared memory (a kernel's first cluster barrier, where there was none).
template <typename Stage, typename Started>
__device__ __forceinline__ int km_cluster(const KmView& kv, const KmParams& p,
                                          cg::cluster_group& cluster, Stage stage,
                                          Started started) {
  KmShared& sh = *kv.sh;
  const KmClLayout& k = kv.k;
  const int R = (int)cluster.num_blocks(), rank = (int)cluster.block_rank();
  const int N = p.N, K = p.K, C = p.C, LK = p.L * p.K, W = (LK + 3) >> 2;
  const int CW = (C + 1) >> 1, CWp = km_cwp(C), NP = k.NP, us = k.us, qs = k.qs, CWc = k.CWc;
  const int tid = threadIdx.x, nthr = blockDim.x, lane = tid & 31, warp = tid >> 5;
  const int nwarps = nthr >> 5;
  const unsigned full = 0xffffffffu;
  const int n_lo = N * rank / R, n_hi = N * (rank + 1) / R;  // N * R < 2^31
  const int wb = W * rank / R, nw = W * (rank + 1) / R - wb;  // own words
  const int nu = min(LK, 4 * (wb + nw)) - 4 * wb;             // own users
  int* lab = reinterpret_cast<int*>(kv.base + k.o_lab);
  int* nlab = reinterpret_cast<int*>(kv.base + k.o_nlab);
  int* own = reinterpret_cast<int*>(kv.base + k.o_own);
  int* chg = reinterpret_cast<int*>(kv.base + k.o_chg);
  uint32_t* cnt = reinterpret_cast<uint32_t*>(kv.base + k.o_cnt);
  uint32_t* pw = reinterpret_cast<uint32_t*>(kv.base + k.o_pw);
  uint32_t* in = reinterpret_cast<uint32_t*>(kv.base + k.o_in);
  unsigned long long* qin = reinterpret_cast<unsigned long long*>(kv.base + k.o_q);
  int* S = reinterpret_cast<int*>(kv.base + k.o_s);
  const int in_words = R * us * k.es;  // of one buffer
  auto pilot = [&](int n, int u) { return (int)((pw[(u >> 2) * NP + n] >> (8 * (u & 3))) & 0xffu); };
  if (warp == nwarps - 1) {
    for (int c = lane; c < C; c += 32) {
      DrawStream ds(p.seed, 0, (uint64_t)p.gen, kTagIsland);
      sh.rdraw[c] = below(ds.draw((uint32_t)c), (uint32_t)(N - c));
    }
  } else {
    const int st = nthr - 32;
    stage(pw, NP, wb, nw);
    for (int i = tid; i < 4 * nw * K * CWp; i += st) cnt[i] = 0;
    for (int n = tid; n < N; n += st) {
      chg[n] = n;  // the initial permutation
      lab[n] = -1;
      int r = (n * R) / N;  // the smallest r with n < N (r + 1) / R
      while (n >= N * (r + 1) / R) ++r;
      own[n] = r << 16 | (n - N * r / R);
    }
    if (tid < kMaxIslands) sh.stale[tid] = 1;
  }
  __syncthreads();
  if (tid == 0) {
    for (int c = 0; c < C; ++c) {
      const int j = c + (int)sh.rdraw[c];
      const int t = chg[c];
      chg[c] = chg[j];
      chg[j] = t;
    }
  }
  if (tid < C) sh.m[tid] = 1;
  __syncthreads();
  for (int t = tid; t < C * nu; t += nthr) {  // one-hots of the initial members
    const int c = t / nu, u = t - c * nu;
    atomicAdd(cnt + (u * K + pilot(chg[c], u)) * CWp + (c >> 1), 1u << ((c & 1) * 16));
  }
  // the sums this warp pushes in each pass: its first (member group, split)
  const int G = (N + 31) >> 5, tasks = G * us;
  int fn = -1, fw0 = 0, fw1 = 0;
  uint32_t fto = 0;
  auto task = [&](int t, int& n, int& w0, int& w1, uint32_t& to) {
    const int g = t / us, s = t - g * us;
    n = g * 32 + lane < N ? g * 32 + lane : -1;
    w0 = nw * s / us;
    w1 = nw * (s + 1) / us;
    if (n >= 0) {
      const int o = own[n];
      to = km_mapa(in + (rank * us + s) * k.es + (o & 0xffff) * CWc, o >> 16);
    }
  };
  if (warp < tasks) task(warp, fn, fw0, fw1, fto);
  // a changed member and own user per thread of the updates
  const int nu1 = max(nu, 1), uq = max(1, nthr / nu1), u_first = tid % nu1, q_first = tid / nu1;
  const int lc = 31 - __clz(CWc);  // CWc is a power of two
  const int lp = C > 16 ? 5 : 32 - __clz(C - 1);  // lanes per member when choosing: >= C or 32
  __syncthreads();
  started();
  int passes = 0;
  for (int it = 0; it < p.max_iter; ++it) {
    // ---- 1. sums over the own users, pushed to the members' owners; warps
    // from the last down: the own share of Q, pushed to every CTA
    for (int t = nwarps - 1 - warp; t < CW * qs; t += nwarps) {
      const int i = t % CW, s = t / CW, e1 = nu * K;
      unsigned long long q0 = 0, q1 = 0;
      for (int e = s * 32 + lane; e < e1; e += 32 * qs) {
        const uint32_t v = cnt[e * CWp + i], lo = v & 0xffffu, hi = v >> 16;
        q0 += lo * lo;  // (counts <= 4096)
        q1 += hi * hi;
      }
      q0 = warp_sum_u48(q0);  // (at most 4096 * 64 counts of at most 4096 each)
      q1 = warp_sum_u48(q1);
      if (lane < R) {
        const uint32_t to = km_mapa(qin + (rank * qs + s) * C + 2 * i, lane);
        km_st64(to, q0);
        if (2 * i + 1 < C) km_st64(to + 8, q1);
      }
    }
    for (int i0 = 0, ch = 0; i0 < CW; i0 += CWc, ++ch) {
      for (int t = warp; t < tasks; t += nwarps) {
        int n = fn, w0 = fw0, w1 = fw1;
        uint32_t to = fto;
        if (t != warp) task(t, n, w0, w1, to);
        if (n >= 0) {
          to += (uint32_t)(ch & 1) * 4u * in_words;
          switch (min(CWc, CW - i0)) {
#define PA_KM_CASE(NW)                                                             \
  case NW:                                                                         \
    km_push<NW>(cnt, CWp, K, pw, NP, n, w0, w1, i0, CWc, to);                      \
    break;
            PA_KM_CASE(1)
            PA_KM_CASE(2)
            PA_KM_CASE(3)
            PA_KM_CASE(4)
            PA_KM_CASE(5)
            PA_KM_CASE(6)
            PA_KM_CASE(7)
            default:
              km_push<8>(cnt, CWp, K, pw, NP, n, w0, w1, i0, CWc, to);
#undef PA_KM_CASE
          }
        }
      }
      cluster.sync();
      // the shares of the own slice: a warp a member, lanes over words and shares
      const uint32_t* buf = in + (ch & 1) * in_words;
      const int i = lane & (CWc - 1), c = 2 * (i0 + i), E = R * us;
      for (int nl = warp; nl < n_hi - n_lo; nl += nwarps) {
        int lo = 0, hi = 0;
        for (int e = lane >> lc; e < E; e += 32 >> lc) {
          const uint32_t v = buf[e * k.es + nl * CWc + i];
          lo += (int)(v & 0xffffu);
          hi += (int)(v >> 16);
        }
        for (int off = 16; off >= CWc; off >>= 1) {
          lo += __shfl_xor_sync(full, lo, off);
          hi += __shfl_xor_sync(full, hi, off);
        }
        if (lane < CWc && c < C) {
          S[nl * C + c] = lo;
          if (c + 1 < C) S[nl * C + c + 1] = hi;
        }
      }
    }
    // the totals of Q (warps from the last down)
    for (int c = nwarps - 1 - warp; c < C; c += nwarps) {
      unsigned long long q = 0;
      for (int r = lane; r < R * qs; r += 32) q += qin[r * C + c];
      q = warp_sum_u48(q);
      if (lane == 0) sh.Q[c] = q;
    }
    __syncthreads();
    // ---- 2. nearest centroids of the own slice, labels to every CTA.  A lane
    // a cluster (two above 32), as many members per warp as fit: squared
    // distance A / m^2 by cross-multiplication, ties to the lower cluster.
    auto nearer = [](long long A, int ma, int a, long long B, int mb, int b) {
      const long long x = A * mb * mb, y = B * ma * ma;
      return x < y || (x == y && a < b);
    };
    for (int n0 = warp << (5 - lp); n0 < n_hi - n_lo; n0 += nwarps << (5 - lp)) {
      const int nl = n0 + (lane >> lp), c0 = lane & ((1 << lp) - 1);
      const bool in_slice = nl < n_hi - n_lo;
      int best = -1, bm = 1;
      long long bd = 0;
      for (int c = c0; c < C && in_slice; c += 32) {
        const long long mc = sh.m[c];
        const long long A = (long long)LK * mc * mc - 2 * mc * (long long)S[nl * C + c] +
                            (long long)sh.Q[c];
        if (best < 0 || nearer(A, (int)mc, c, bd, bm, best)) {
          best = c;
          bm = (int)mc;
          bd = A;
        }
      }
      for (int off = (1 << lp) >> 1; off > 0; off >>= 1) {
        const long long od = __shfl_xor_sync(full, bd, off);
        const int om = __shfl_xor_sync(full, bm, off), o = __shfl_xor_sync(full, best, off);
        if (o >= 0 && (best < 0 || nearer(od, om, o, bd, bm, best))) {
          best = o;
          bm = om;
          bd = od;
        }
      }
      if (in_slice)
        for (int r = c0; r < R; r += 1 << lp)
          km_st(km_mapa(nlab + n_lo + nl, r), (uint32_t)best);
    }
    if (tid < kMaxIslands) sh.nm[tid] = 0;
    if (tid == 0) sh.nchg = 0;
    cluster.sync();
    // ---- 3. changed members and sizes; every CTA finds the same
    for (int n0 = warp * 32; n0 < N; n0 += nthr) {
      const int n = n0 + lane;
      const bool valid = n < N;
      const int nl = valid ? nlab[n] : -1 - lane, old = valid ? lab[n] : nl;
      const bool moved = nl != old;
      const unsigned bm = __ballot_sync(full, moved);
      if (bm) {
        const int leader = __ffs(bm) - 1;
        int at = 0;
        if (lane == leader) at = atomicAdd(&sh.nchg, __popc(bm));
        at = __shfl_sync(full, at, leader);
        if (moved) chg[at + __popc(bm & ((1u << lane) - 1u))] = (n << 13) | ((old + 1) << 6) | nl;
      }
      const unsigned same = __match_any_sync(full, nl);
      if (valid) {
        lab[n] = nl;
        if ((int)(__ffs(same) - 1) == lane) atomicAdd(&sh.nm[nl], __popc(same));
      }
    }
    __syncthreads();
    ++passes;
    const int total = sh.nchg;
    if (total == 0 || it == p.max_iter - 1) break;
    // clusters that gain members after having none restart at zero
    bool any = false;
    for (int c = lane; c < C; c += 32) any |= sh.stale[c] && sh.nm[c] > 0;
    if (__any_sync(full, any)) {  // (the same in every warp)
      for (int e = tid; e < nu * K; e += nthr)
        for (int i = 0; i < CW; ++i) {
          const bool z0 = sh.stale[2 * i] && sh.nm[2 * i] > 0;
          const bool z1 = 2 * i + 1 < C && sh.stale[2 * i + 1] && sh.nm[2 * i + 1] > 0;
          if (z0 || z1) cnt[e * CWp + i] &= (z0 ? 0u : 0xffffu) | (z1 ? 0u : 0xffff0000u);
        }
      __syncthreads();
    }
    if (tid < C && sh.nm[tid] > 0) sh.m[tid] = sh.nm[tid];
    // every changed member's one-hot moves from its old cluster (when that one
    // still has members) to its new one, for the own users
    auto move = [&](int q, int u) {
      const int e = chg[q], n = e >> 13, A = ((e >> 6) & 127) - 1, B = e & 63;
      uint32_t* row = cnt + (u * K + pilot(n, u)) * CWp;
      atomicAdd(row + (B >> 1), 1u << ((B & 1) * 16));
      if (A >= 0 && sh.nm[A] > 0)  // (the half is >= 1: no borrow)
        atomicAdd(row + (A >> 1), 0u - (1u << ((A & 1) * 16)));
    };
    if (nu <= nthr) {
      if (tid < uq * nu)
        for (int q = q_first; q < total; q += uq) move(q, u_first);
    } else {
      for (int q = 0; q < total; ++q)
        for (int u = tid; u < nu; u += nthr) move(q, u);
    }
    __syncthreads();
    if (tid < C) sh.stale[tid] = sh.nm[tid] == 0;
  }
  return passes;
}

}  // namespace
}  // namespace pa
