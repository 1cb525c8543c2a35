// Helpers shared by the two bucket-join kernels (join.cu, and the tcgen05 form in
// join_tc.cu): the top-k insertion network, the view of one image's bucket-sorted
// table, the per-pair Hamming threshold, the finalisation of a pair's survivor
// lists, and the launch sizes.
#pragma once

#include <cuda_fp16.h>

#include "internal.h"

namespace chx {

constexpr int JT = 256;  // threads of a CTA of the tcgen05 form

// Insertion that drops a key equal to one already kept.
template <int KC>
__device__ __forceinline__ void jt_insert(uint32_t (&top)[KC], uint32_t k) {
#pragma unroll
  for (int s = 0; s < KC; ++s) {
    const uint32_t t = top[s];
    const bool dup = (t == k);
    top[s] = min(t, k);
    k = dup ? KEY_INF : max(t, k);
  }
}

// Insertion that keeps equal keys (side by side): two independent operations per entry.
template <int KN>
__device__ __forceinline__ void jt_insert_any(uint32_t (&top)[KN], uint32_t k) {
#pragma unroll
  for (int s = KN - 1; s > 0; --s) top[s] = max(top[s - 1], min(top[s], k));
  top[0] = min(top[0], k);
}

// The K-th smallest (K <= KC) of a sorted list.
template <int KC, int KN>
__device__ __forceinline__ uint32_t jt_kth(const uint32_t (&top)[KN], uint32_t K) {
  uint32_t v = KEY_INF;
#pragma unroll
  for (int s = 0; s < KC; ++s)
    if ((uint32_t)s + 1 == K) v = top[s];
  return v;
}

__device__ __forceinline__ uint32_t jt_hamming(uint4 a, uint4 b) {
  return __popc(a.x ^ b.x) + __popc(a.y ^ b.y) + __popc(a.z ^ b.z) + __popc(a.w ^ b.w);
}

struct JView {  // one image's bucket-sorted table t
  const uint32_t* off;
  const uint32_t* idx;
  const uint4* rec;
};

__device__ __forceinline__ JView jview(const uint8_t* join, uint64_t base, uint32_t n, uint32_t t) {
  const uint8_t* b = join + base + (uint64_t)t * join_block(n);
  JView v;
  v.off = reinterpret_cast<const uint32_t*>(b);
  v.idx = reinterpret_cast<const uint32_t*>(b + 1040);
  v.rec = reinterpret_cast<const uint4*>(b + 1040 + 4 * ((n + 3) / 4 * 4));
  return v;
}

// Hamming threshold for a pair: the 99.5th percentile of the k-th distances
// seen so far (histogram kept across launches), else the calibration / host
// hint; 0 = none.  Computed by warp 0.
__device__ __forceinline__ uint32_t pair_threshold(const MatchArgs& a, uint32_t p, int lane) {
  const uint32_t* h = a.jhist + (size_t)p * HBINS;
  uint32_t v[5], tot = 0;
#pragma unroll
  for (int k = 0; k < 5; ++k) {
    const uint32_t b = lane * 5 + k;  // lanes own 5 consecutive bins
    v[k] = b < HBINS ? *reinterpret_cast<const volatile uint32_t*>(h + b) : 0u;
    tot += v[k];
  }
  uint32_t incl = tot;
#pragma unroll
  for (int d = 1; d < 32; d <<= 1) {
    const uint32_t o = __shfl_up_sync(0xFFFFFFFFu, incl, d);
    if (lane >= d) incl += o;
  }
  const uint32_t all = __shfl_sync(0xFFFFFFFFu, incl, 31);
  uint32_t guess = *reinterpret_cast<const volatile uint32_t*>(a.tau_pair + p);
  if (!a.tau_fixed && all >= 64) {
    const uint32_t want = all - all / 200;  // 99.5 %
    uint32_t run = incl - tot, bin = 0xFFFFFFFFu;
#pragma unroll
    for (int k = 0; k < 5; ++k) {
      run += v[k];
      if (bin == 0xFFFFFFFFu && run >= want) bin = lane * 5 + k;
    }
    uint32_t best = bin;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) best = min(best, __shfl_xor_sync(0xFFFFFFFFu, best, o));
    if (best != 0xFFFFFFFFu) guess = best + 1u;
  }
  return guess;
}

// Words per query of the finalisation's keys and distances.
__host__ __device__ constexpr int join_kp(int KC) { return (KC + 3) / 4 * 4; }

// The K <= KC smallest distinct keys of a survivor list of m <= JSEG entries, ascending, then KEY_INF, to keys[KC].
// Not inlined: the finalisation's own pass would pay for its registers.
template <int KC>
__device__ __noinline__ void jt_distinct(const uint32_t* list, uint32_t m, uint32_t K, uint32_t* keys) {
  uint32_t top[KC];
#pragma unroll
  for (int s = 0; s < KC; ++s) top[s] = KEY_INF;
#pragma unroll 1
  for (uint32_t e0 = 0; e0 < m; e0 += 4) {
    const uint4 x = __ldcg(reinterpret_cast<const uint4*>(list) + e0 / 4);  // (the list has JSEG entries)
    const uint32_t kk[4] = {x.x, x.y, x.z, x.w};
#pragma unroll
    for (int u = 0; u < 4; ++u)
      if (e0 + u < m && kk[u] < top[KC - 1]) jt_insert<KC>(top, kk[u]);
  }
#pragma unroll
  for (int s = 0; s < KC; ++s) keys[s] = (uint32_t)s < K ? top[s] : KEY_INF;
}

// Whether a query meets most of its candidates in several tables, so that the finalisation reads its list by
// jt_distinct at once.  us per pass over 400 pairs, 6 tables, after a pass that keeps repeats / at once: 6,000 x 6,000
// features, 7 bits k = 10 1,524 / 1,513, k = 16 2,060 / 2,014; 6 bits 2,002 / 1,930 and 3,112 / 2,717; 4 bits, k = 10
// 9,724 / 9,162; 1,000 x 1,000, 7 bits k = 32 1,023 / 858.  With 8 bits few queries have repeats beyond the spare entries.
__host__ __device__ inline bool join_repeats(const KParams& kp) { return kp.n_tables > 1 && kp.bits_per_table <= 7; }

// Finalisation of up to 32 queries of a pair by one warp, the lane's query q (valid: it exists) with n keys
// counted in its survivor list: the k smallest distinct survivors (Step 3), exact squared distances of those k
// with 4 lanes per 128-byte row (Step 4, Sec. 5.2) and Lowe's ratio test.  A query whose list overflowed, or
// that holds fewer than k survivors while the guess may have turned a candidate away (cut), is left PENDING for
// the exact fallback.  key_s, dist_s: 32 join_kp(KC) words each, the warp's own.
// Bound by issue: the insertion network keeps equal keys (two independent operations per entry instead of four
// dependent ones; repeats are dropped once at the end, and where that loses keys, or would for most queries, the list
// is read by jt_distinct) and the distances take 67 instructions per four rows of
// eight queries (one exchange tree for four sums).  Per 32 queries about 3,100 warp instructions, 4,500 before.
// Queries that lose keys to repeats are not left to the fallback: with that, 400 pairs of 1,000 x 1,000 features, 8
// tables of 4 bits, k = 10 took 1,140 us a pass, now 570; 6,000 x 6,000 25.5 ms, now 12.2; images of near copies of
// each descriptor, 6 tables of 8 bits, 6,000 x 6,000 3,745 us, now 1,663.
template <int KC, bool EPI>
__device__ __forceinline__ void finalise_warp(const MatchArgs& a, const PairInfo& P, uint32_t it, bool cut, uint32_t q,
                                              bool valid, uint32_t n, const uint32_t* list, uint32_t* key_s,
                                              uint32_t* dist_s, uint32_t* s_hist) {
  const KParams& kp = a.kp;
  const uint32_t T = kp.n_tables, K = kp.top_k;
  constexpr int KN = KC + 2;  // two more than the instantiation's k: room for repeated keys
  constexpr int KP = join_kp(KC);
  const int lane = threadIdx.x & 31;
  uint32_t top[KN];
#pragma unroll
  for (int s = 0; s < KN; ++s) top[s] = KEY_INF;
  bool pending = false, again = join_repeats(kp);  // again: the keys come from jt_distinct
  if (valid) {
    pending = n > JSEG;  // survivors were dropped
    const uint4* ql = reinterpret_cast<const uint4*>(list);
    const uint32_t m = again ? 0u : min(n, JSEG);
    // a key at or above the list's last entry when its group of eight starts cannot enter it
    for (uint32_t e0 = 0; e0 < m; e0 += 8) {
      const uint4 x0 = __ldcg(ql + e0 / 4), x1 = __ldcg(ql + e0 / 4 + 1);  // (the list has JSEG entries)
      const uint32_t lim = top[KN - 1], kk[8] = {x0.x, x0.y, x0.z, x0.w, x1.x, x1.y, x1.z, x1.w};
#pragma unroll
      for (int u = 0; u < 8; ++u)
        if (e0 + u < m && kk[u] < lim && kk[u] != top[0]) jt_insert_any<KN>(top, kk[u]);
    }
    // drop the repeated keys that are left (adjacent now); a full list that lost more than two may miss a key
    bool rep = false;
#pragma unroll
    for (int s = 1; s < KN; ++s) rep |= top[s] == top[s - 1] && top[s] != KEY_INF;
    if (rep) {
      const bool full = top[KN - 1] != KEY_INF;
      for (int r = 0; r + 1 < KN; ++r) {
        bool seen = false;  // removes the first repeated key
#pragma unroll
        for (int s = 1; s < KN; ++s) {
          seen |= top[s] == top[s - 1] && top[s] != KEY_INF;
          if (seen) top[s] = s + 1 < KN ? top[s + 1 < KN ? s + 1 : s] : KEY_INF;
        }
        if (!seen) break;
      }
      again = full && jt_kth<KC>(top, K) == KEY_INF;
    }
  }
  again = again && valid && !pending;
  uint32_t* keys = key_s + lane * KP;
#pragma unroll
  for (int s = 0; s < KP; s += 4) {
    const bool ok = valid && !pending;
    uint4 k4;
    k4.x = ok && (uint32_t)s < K ? top[s] : KEY_INF;
    k4.y = ok && (uint32_t)s + 1 < K ? top[s + 1 < KN ? s + 1 : 0] : KEY_INF;
    k4.z = ok && (uint32_t)s + 2 < K ? top[s + 2 < KN ? s + 2 : 0] : KEY_INF;
    k4.w = ok && (uint32_t)s + 3 < K ? top[s + 3 < KN ? s + 3 : 0] : KEY_INF;
    *reinterpret_cast<uint4*>(keys + s) = k4;
  }
  if (__any_sync(0xFFFFFFFFu, again)) {  // (top is not needed any more: a call here costs the others nothing)
    if (again) jt_distinct<KC>(list, n, K, keys);
  }
  if (valid) {
    const uint32_t kth = keys[K - 1];
    if (!pending && kth == KEY_INF && cut) {
      // fewer than k: exact only if no candidate was turned away by the guess
      const uint2 qbk = __ldg(reinterpret_cast<const uint2*>(a.buckets) + P.a0 + q);
      uint32_t nlook = 0;
      for (uint32_t t = 0; t < T; ++t) {
        const JView B = jview(a.join, P.bjoin, P.nB, t);
        const uint32_t v = (t < 4 ? (qbk.x >> (8 * t)) : (qbk.y >> (8 * (t - 4)))) & 0xFFu;
        nlook += __ldg(B.off + v + 1) - __ldg(B.off + v);
      }
      pending = nlook > n;
      if (pending)
        for (uint32_t s = 0; s < K; ++s) keys[s] = KEY_INF;
    }
    if (!EPI && !pending && kth != KEY_INF && !a.tau_fixed) atomicAdd(s_hist + (kth >> 24), 1u);
  }
  __syncwarp();
  // 4 lanes per 128-byte row (32 bytes each), 8 queries per step, four candidates' rows in flight; a missing
  // candidate reads the image's first row.  The four dot products are summed over the four lanes by three
  // exchanges, which leave candidate s + sub's sum in lane sub.
  const int grp = lane >> 2, sub = lane & 3;
  const uint8_t* bd = a.desc + P.b0 * DIM + 32 * sub;
  const uint32_t* bsq = a.sqnorm + P.b0;
  for (int qq0 = 0; qq0 < 32 && P.nB; qq0 += 8) {
    const int qi = qq0 + grp;
    const uint32_t qg = min(__shfl_sync(0xFFFFFFFFu, q, qi), P.nA - 1);
    const uint4* arow = reinterpret_cast<const uint4*>(a.desc + (P.a0 + qg) * DIM + 32 * sub);
    const uint4 a0 = __ldg(arow), a1 = __ldg(arow + 1);
    const uint32_t sa = __ldg(a.sqnorm + P.a0 + qg);
#pragma unroll 1
    for (uint32_t s = 0; s < K; s += 4) {
      const uint4 key = *reinterpret_cast<const uint4*>(key_s + qi * KP + s);
      const uint32_t kk[4] = {key.x, key.y, key.z, key.w};
      uint4 b0[4], b1[4];
      uint32_t jj[4], dot[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        jj[u] = kk[u] == KEY_INF ? 0u : kk[u] & 0xFFFFFFu;
        const uint4* brow = reinterpret_cast<const uint4*>(bd + (size_t)jj[u] * DIM);
        b0[u] = __ldg(brow);
        b1[u] = __ldg(brow + 1);
      }
      const uint32_t jm = sub & 2 ? (sub & 1 ? jj[3] : jj[2]) : (sub & 1 ? jj[1] : jj[0]);
      const uint32_t sb = __ldg(bsq + jm);
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        dot[u] = __dp4a(a0.x, b0[u].x, 0u);
        dot[u] = __dp4a(a0.y, b0[u].y, dot[u]);
        dot[u] = __dp4a(a0.z, b0[u].z, dot[u]);
        dot[u] = __dp4a(a0.w, b0[u].w, dot[u]);
        dot[u] = __dp4a(a1.x, b1[u].x, dot[u]);
        dot[u] = __dp4a(a1.y, b1[u].y, dot[u]);
        dot[u] = __dp4a(a1.z, b1[u].z, dot[u]);
        dot[u] = __dp4a(a1.w, b1[u].w, dot[u]);
      }
      // lanes 0, 1 keep candidates 0, 1 and lanes 2, 3 candidates 2, 3; then even / odd
      const bool hi = sub & 2, od = sub & 1;
      const uint32_t x0 = (hi ? dot[2] : dot[0]) + __shfl_xor_sync(0xFFFFFFFFu, hi ? dot[0] : dot[2], 2);
      const uint32_t x1 = (hi ? dot[3] : dot[1]) + __shfl_xor_sync(0xFFFFFFFFu, hi ? dot[1] : dot[3], 2);
      const uint32_t d = (od ? x1 : x0) + __shfl_xor_sync(0xFFFFFFFFu, od ? x0 : x1, 1);
      dist_s[qi * KP + s + sub] = sa + sb - 2u * d;
    }
  }
  __syncwarp();
  bool matched = false;
  if (valid) {
    uint32_t nv = 0, d1 = 0xFFFFFFFFu, d2 = 0xFFFFFFFFu, j1 = NO_MATCH;
#pragma unroll
    for (int s = 0; s < KP; s += 4) {
      if ((uint32_t)s >= K) break;
      const uint4 k4 = *reinterpret_cast<const uint4*>(key_s + lane * KP + s);
      const uint4 d4 = *reinterpret_cast<const uint4*>(dist_s + lane * KP + s);
      const uint32_t kk[4] = {k4.x, k4.y, k4.z, k4.w}, dd[4] = {d4.x, d4.y, d4.z, d4.w};
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const bool is = kk[u] != KEY_INF;
        const uint32_t d = is ? dd[u] : 0xFFFFFFFFu, jx = kk[u] & 0xFFFFFFu;
        nv += is ? 1u : 0u;
        const bool first = is && (d < d1 || (d == d1 && jx < j1));
        d2 = first ? d1 : min(d2, d);
        j1 = first ? jx : j1;
        d1 = first ? d : d1;
      }
    }
    matched = ratio_ok(kp, nv, d1, d2);
    a.res[P.qbase + q] = pending ? PENDING : (matched ? j1 : NO_MATCH);
  }
  const uint32_t bal = __ballot_sync(0xFFFFFFFFu, matched);
  if (lane == 0 && bal) atomicAdd(a.pair_cnt + it, (unsigned long long)__popc(bal));
  __syncwarp();
}

// The same for all queries of a pair by a CTA of JT threads, whose counters cnt_s holds.
template <int KC, bool EPI>
__device__ __forceinline__ void join_finalise(const MatchArgs& a, const PairInfo& P, uint32_t it, bool cut,
                                              const uint32_t* cnt_s, const uint32_t* seg, uint32_t* key_s,
                                              uint32_t* dist_s, uint32_t* s_hist) {
  const uint32_t w = threadIdx.x / 32 * 32 * join_kp(KC);
  for (uint32_t q0 = 0; q0 < P.nA; q0 += JT) {
    const uint32_t q = q0 + threadIdx.x;
    finalise_warp<KC, EPI>(a, P, it, cut, q, q < P.nA, q < P.nA ? cnt_s[q] : 0u, seg + (size_t)q * JSEG, key_s + w,
                           dist_s + w, s_hist);
  }
}

// Instantiation (keys kept per query) for k.
inline int join_kc(uint32_t k) { return k <= 4 ? 4 : k <= 8 ? 8 : k <= 10 ? 10 : k <= 16 ? 16 : 32; }

// Resident CTAs of a join kernel for n_items pairs (at most ctas_per_sm per SM when non-zero); 0 when its
// shared memory does not fit.  Raises the kernel's shared-memory limit on the current device.
inline uint32_t join_resident(void (*kern)(MatchArgs), size_t smem, uint32_t n_items, uint32_t ctas_per_sm,
                              int threads = JT) {
  int dev = 0, nsm = 0, optin = 0, occ = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
  cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
  if (smem + 4096 > (size_t)optin) return 0;
  if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, optin - 2048) != cudaSuccess ||
      cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, kern, threads, smem) != cudaSuccess || occ < 0) {
    cudaGetLastError();
    occ = 0;
  }
  if (ctas_per_sm && ctas_per_sm < (uint32_t)occ) occ = (int)ctas_per_sm;
  const uint64_t gr = (uint64_t)nsm * (uint64_t)occ;
  return (uint32_t)(n_items < gr ? n_items : gr);
}

}  // namespace chx
