// Batched matching as a bucket join: Steps 1-4 of Sec. 3.1 (+ the Sec. 6
// threshold tau, + the Sec. 7.2 band) organised around the lookup tables.
//
// Step 1 pairs a query with exactly the candidates that share its bucket in
// some table, so for table t and short code v the work is the dense block
// (queries of A in bucket v) x (candidates of B in bucket v).  A warp takes one
// block from the bucket-sorted tables (codes stored inline): the candidates are
// staged in shared memory, every lane holds one query's 128-bit code, and a step
// gives all 32 lanes the Hamming distance (Step 2) to one candidate.  Keys
// H << 24 | j with H <= theta (theta: the pair's threshold guess, learned per
// pair from the k-th distances of earlier launches, capped by the Sec. 6 tau) go
// to the query's survivor list: a counter per query in shared memory, JSEG
// entries per query in global memory.  The scan takes one table after the other,
// with a barrier between them: a query lies in one bucket of a table, so within a
// table its list has a single writer, and the lane keeps the position in a
// register.  Then the CTA finalises the pair's queries (join_common.cuh).  A
// query whose list overflowed, or that holds fewer than k distinct survivors
// while the guess turned some candidate away, is left PENDING for the exact
// fallback kernel, so results never depend on the guess.  A list counts as
// overflowed once fewer than four of its slots are left and its query meets
// further candidates: a step takes four of them without a test per store.  Filled
// to the last slot instead, us per pass over 400 pairs of 6,000 x 6,000 features: 8
// bits, k = 2 892 -> 917, 6 tables of 4 bits, k = 2 5,215 -> 5,476, k = 16 26,369 ->
// 24,673.
//
// With the band (EPI) a candidate outside it is no candidate at all, so there is
// no Hamming guess, and the band test, cheaper than a Hamming distance and passed
// by few, comes first.
//
// Why the distances are population counts and not a tensor-core contraction: on
// sm_103a an FP8 mma.sync executes as two tensor instructions after converting
// its operands, and expanding codes to +-1 operands, converting them and moving
// each survivor out of the accumulator layout cost more instructions than the
// counts they replace.  Per lookup entry (500 pairs of 8k x 8k features): 2.40
// warp instructions with FP8 mma.sync in 16 x 32 blocks (35 % of their slots were
// entries), 1.60 here.  f16 operands that hold two code bits each (four MMAs per
// 16 x 8 tile, exact in f32 accumulators) took 20.6 ms on the 4,950 pairs below.
// What bounds the kernel now is memory latency and issue (56 % of the slots; half
// of the stalls wait for tables, lists and rows): with two CTAs of 512 threads
// per SM the lists of the pairs in flight (about 1.2 MB each) exceed the L2 (a
// timing copy whose lists fit it: 8.9 ms instead of 14 for the scan).  4,950
// pairs of 8k x 8k: 25.0 -> 16.8 ms; 11,527 uneven pairs (1,000 to 20,000
// features): 52.9 -> 31.6 ms.
#include <cooperative_groups.h>

#include "join_common.cuh"

namespace chx {

namespace cg = cooperative_groups;

constexpr int CAL_SAMPLES = 128;   // calibration: sampled queries per pair
constexpr uint32_t CAL_MARGIN = 1; // calibration: Hamming margin over the second largest sample

// ---------------------------------------------------------------------------
// The scan of one (table, bucket) block by one warp.
// ---------------------------------------------------------------------------
constexpr int JNT = 512;       // threads of a CTA (two per SM; 4 x 256: 17.3 ms, 1 x 1024: 16.9 against 16.7)
constexpr uint32_t JCOL = 64;  // candidates of a bucket staged in shared memory at a time, per warp

// Shared memory of a warp: the staged candidates' codes and indices, and with the band their key-points.
template <bool EPI>
struct JoinWarp {
  uint4 col[JCOL];
  uint32_t colj[JCOL];
};
template <>
struct JoinWarp<true> : JoinWarp<false> {
  float2 colp[JCOL];
};

// The 2^lg CTAs of a cluster share a pair: 32 queries at a time, tile q / 32 belongs to CTA (q / 32) % 2^lg,
// which holds the queries' survivor counters (a byte each) and finalises them.
__host__ __device__ inline uint32_t join_own(uint32_t na, uint32_t lg) {
  return (((na + 31) / 32 + (1u << lg) - 1) >> lg) * 32;
}
// Shared memory of a CTA: its counters, then the warps' parts and the bucket offsets ([2][T][2^m + 1]), or the
// finalisation's keys and distances.
__host__ __device__ inline size_t join_smem_bytes(int KC, uint32_t T, uint32_t na_max, uint32_t lg, bool epi) {
  const size_t fin = (size_t)2 * join_kp(KC) * JNT * 4,
               scan = (JNT / 32) * (epi ? sizeof(JoinWarp<true>) : sizeof(JoinWarp<false>)) + (size_t)2 * T * 257 * 4;
  return join_own(na_max, lg) + (fin > scan ? fin : scan);
}

template <bool CL>
struct JoinLists {
  uint32_t* seg;   // [queries][JSEG] survivors' keys, in global memory
  uint8_t* cnt_s;  // this CTA's counters
  uint32_t lg;
  __device__ __forceinline__ uint8_t* count(uint32_t q) const {
    if constexpr (!CL) return cnt_s + q;
    const uint32_t t = q / 32;
    return cg::this_cluster().map_shared_rank(cnt_s, t & ((1u << lg) - 1u)) + ((t >> lg) * 32 + q % 32);
  }
};

// popc(x) + popc(y) + popc(z) + popc(w) with three population counts (a carry-save step on x, y, z).
__device__ __forceinline__ uint32_t popc128(uint32_t x, uint32_t y, uint32_t z, uint32_t w) {
  const uint32_t s = x ^ y ^ z, c = (x & y) | (z & (x | y));
  return __popc(s) + __popc(w) + 2 * __popc(c);
}

// Four candidates for the 32 lanes' queries: the keys H << 24 | j of the survivors (H <= h_thr, the first n of
// the four) go to the lane's next list slots (byte offset off from list), by predicate: survivors are
// scattered over lanes and steps, and a branch per step would diverge.
template <bool TAIL>
__device__ __forceinline__ void scan4(uint4 q, uint32_t& off, int h_thr, const uint4* col, const uint32_t* colj,
                                      uint32_t n, uint64_t list) {
  uint4 c[4];
  uint32_t j[4], h[4];
#pragma unroll
  for (int u = 0; u < 4; ++u) {
    c[u] = col[u];
    j[u] = colj[u];
  }
#pragma unroll
  for (int u = 0; u < 4; ++u) {
    h[u] = popc128(q.x ^ c[u].x, q.y ^ c[u].y, q.z ^ c[u].z, q.w ^ c[u].w);
    j[u] += h[u] << 24;
  }
#pragma unroll
  for (int u = 0; u < 4; ++u)
    asm volatile(
        "{\n .reg .pred p;\n .reg .u64 d;\n setp.le.s32 p, %1, %2;\n mad.wide.u32 d, %0, 1, %4;\n"
        " @p st.global.u32 [d], %3;\n @p add.u32 %0, %0, 4;\n}"
        : "+r"(off)
        : "r"(h[u]), "r"(!TAIL || (uint32_t)u < n ? h_thr : -1), "r"(j[u]), "l"(list)
        : "memory");
}

// The queries qs .. qs + nq of A's bucket against the nb staged candidates.
template <bool CL>
__device__ __forceinline__ void scan_rows(const JoinWarp<false>& w, const JView& A, uint32_t qs, uint32_t nq, uint32_t nb,
                                          uint32_t h_thr, const JoinLists<CL>& L, int lane) {
  for (; nq > 16; qs += min(nq, 32u), nq -= min(nq, 32u)) {
    if ((uint32_t)lane < nq) {
      const uint4 code = __ldg(A.rec + qs + lane);
      const uint32_t q = __ldg(A.idx + qs + lane);
      const uint64_t list = (uint64_t)__cvta_generic_to_global(L.seg + (size_t)q * JSEG);
      uint8_t* cnt = L.count(q);
      uint32_t off = 4u * *cnt, c = 0;  // 4 (JSEG + 1): the list has run out (the query is left PENDING)
#pragma unroll 1
      for (; c < nb; c += 4) {
        const bool room = off <= 4 * (JSEG - 4);
        const int th = room ? (int)h_thr : -1;
        if (c + 4 <= nb) scan4<false>(code, off, th, w.col + c, w.colj + c, 4, list);
        else scan4<true>(code, off, th, w.col + c, w.colj + c, nb - c, list);
        if (!room) off = 4 * (JSEG + 1);
      }
      *cnt = (uint8_t)(off / 4);
    }
    __syncwarp();
  }
  if (nq) {
    // few queries left: S lanes per query, each taking every S-th candidate
    const uint32_t sl = min(4u, (uint32_t)__clz(nq - 1) - 27u), S = 1u << sl;
    const uint32_t k = (uint32_t)lane >> sl, sub = (uint32_t)lane & (S - 1);
    const uint32_t grp = (0xFFFFFFFFu >> (32 - S)) << ((uint32_t)lane - sub), lt = (1u << lane) - 1u;
    uint4 code = make_uint4(0u, 0u, 0u, 0u);
    uint32_t q = 0, n = 0;
    if (k < nq) {
      code = __ldg(A.rec + qs + k);
      q = __ldg(A.idx + qs + k);
      n = *L.count(q);
    }
    uint32_t* list = L.seg + (size_t)q * JSEG;
    for (uint32_t c = sub; c < nb + sub; c += S) {
      uint32_t h = 255u, j = 0;
      if (k < nq && c < nb) {
        const uint4 x = w.col[c];
        j = w.colj[c];
        h = popc128(code.x ^ x.x, code.y ^ x.y, code.z ^ x.z, code.w ^ x.w);
      }
      const uint32_t bal = __ballot_sync(0xFFFFFFFFu, h <= h_thr) & grp;
      const uint32_t pos = n + __popc(bal & lt);
      if (h <= h_thr && pos < JSEG) list[pos] = (h << 24) + j;
      n += __popc(bal);
    }
    if (k < nq && sub == 0) *L.count(q) = (uint8_t)min(n, JSEG + 1u);
    __syncwarp();
  }
}

// The same inside the band of Sec. 7.2: a candidate counts when its distance from the query's epipolar line is
// inside the band and H <= h_thr (tau).  Few candidates do, so 32 at a time take two FMAs and a compare with the
// line's upper threshold (band_line), and the lane's bits that are left take the rest: the lower threshold,
// the FP64 expression in between, the Hamming distance and the store.
// The distance comes last since the band turns nearly all away; with FP8 mma.sync blocks, whose distances come for
// all, and the band test on every slot of the padded blocks, it took 2.72 warp instructions per entry against 0.90.
// 300 pairs of views with about 8,000 key-points: 2.43 -> 0.79 ms; all overlapping pairs of 160 such views:
// 26.9 -> 9.0 ms.  Bound by issue (54 % of the slots, 23 of 32 threads in an instruction) and latency.
struct BandRows {
  const float4* line;  // per query: FP32 a, b, c and the lower threshold on |a x' + b y' + c|
  const float* hi;     // ... and the upper one
  const double* F;
  const float2* kpa;   // key-points of the query image
  double dd;
};
template <bool CL>
__device__ __forceinline__ void scan_rows_band(const JoinWarp<true>& w, const JView& A, uint32_t qs, uint32_t nq,
                                               uint32_t nb, uint32_t h_thr, const JoinLists<CL>& L, const BandRows& R,
                                               int lane) {
  for (uint32_t r0 = 0; r0 < nq; r0 += 32) {
    if (r0 + lane < nq) {
      const uint4 code = __ldg(A.rec + qs + r0 + lane);
      const uint32_t q = __ldg(A.idx + qs + r0 + lane);
      const float4 l = __ldcg(R.line + q);
      const float hi = __ldcg(R.hi + q);
      uint32_t* list = L.seg + (size_t)q * JSEG;
      uint8_t* cnt = L.count(q);
      uint32_t n = *cnt;
#pragma unroll 1
      for (uint32_t c0 = 0; c0 < nb; c0 += 32) {
        uint32_t m = 0;
#pragma unroll
        for (uint32_t u = 0; u < 32; u += 8) {
          if (c0 + u >= nb) break;  // (the last eight may read past nb: masked below)
#pragma unroll
          for (uint32_t e = 0; e < 8; ++e) {
            const float2 p = w.colp[c0 + u + e];
            const float d = fabsf(fmaf(l.x, p.x, fmaf(l.y, p.y, l.z)));
            if (!(d >= hi)) m |= 1u << (u + e);
          }
        }
        if (nb - c0 < 32) m &= (1u << (nb - c0)) - 1u;
        while (m) {
          const uint32_t c = c0 + __ffs(m) - 1;
          m &= m - 1;
          const float2 p = w.colp[c];
          const uint32_t h = jt_hamming(w.col[c], code);
          if (h > h_thr) continue;
          if (!(fabsf(fmaf(l.x, p.x, fmaf(l.y, p.y, l.z))) <= l.w) && !epi_keep_fp64_F(R.F, __ldg(R.kpa + q), R.dd, p))
            continue;
          if (n < JSEG) list[n] = (h << 24) + w.colj[c];
          ++n;
        }
      }
      *cnt = (uint8_t)min(n, JSEG + 1u);
    }
    __syncwarp();
  }
}

template <int KC, bool CL, bool EPI>
__global__ void __launch_bounds__(JNT, 2) k_join(MatchArgs a) {
  extern __shared__ __align__(16) uint8_t jsm[];
  __shared__ uint32_t s_item, s_tau, s_task[CASHASH_MAX_TABLES];
  cg::cluster_group cl = cg::this_cluster();
  const uint32_t lg = CL ? 31u - __clz(cl.num_blocks()) : 0u, rank = CL ? cl.block_rank() : 0u;
  auto sync = [&] {
    if constexpr (CL) cl.sync();
    else __syncthreads();
  };
  __shared__ uint32_t s_hist[HBINS];
  __shared__ PairInfo s_P;
  __shared__ JView s_A[CASHASH_MAX_TABLES], s_B[CASHASH_MAX_TABLES];
  const KParams kp = a.kp;
  const uint32_t T = kp.n_tables, nbk = 1u << kp.bits_per_table;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  uint8_t* cnt_s = jsm;
  uint8_t* work = jsm + join_own(a.na_max, lg);
  JoinWarp<EPI>& w = reinterpret_cast<JoinWarp<EPI>*>(work)[warp];
  uint32_t* off_s = reinterpret_cast<uint32_t*>(reinterpret_cast<JoinWarp<EPI>*>(work) + JNT / 32);
  uint32_t* key_s = reinterpret_cast<uint32_t*>(work);
  uint32_t* dist_s = key_s + join_kp(KC) * JNT;
  const JoinLists<CL> L{a.jqueue + (size_t)(blockIdx.x >> lg) * a.na_max * JSEG, cnt_s, lg};
  const uint32_t* item0 = CL ? cl.map_shared_rank(&s_item, 0) : &s_item;
  uint32_t* task0 = CL ? cl.map_shared_rank(s_task, 0) : s_task;
  const uint32_t h_user = kp.tau < kp.code_bits ? kp.tau : 128u;  // Sec. 6: keys with H > tau are no candidates
  __shared__ uint32_t s_kx, s_ky;  // band: the largest |x'|, |y'| of the candidate image
  float4* lines = EPI ? a.jline + (size_t)(blockIdx.x >> lg) * jline_stride(a.na_max) : nullptr;
  float* lhi = EPI ? reinterpret_cast<float*>(lines + a.na_max) : nullptr;
  const double dd = kp.epi_px * kp.epi_px;
  const uint32_t nbo = T * (nbk + 1), nsp = kp.bits_per_table < 6 ? 6 - kp.bits_per_table : 0;

  for (;;) {
    sync();  // the previous pair is done
    if (rank == 0 && tid == 0) {
      const uint32_t it0 = atomicAdd(a.item_ctr, 1u);
      s_item = it0 < a.n_items ? a.items[it0].x : 0xFFFFFFFFu;
    }
    if (rank == 0 && tid < CASHASH_MAX_TABLES) s_task[tid] = 0;
    for (uint32_t b = tid; b < HBINS; b += JNT) s_hist[b] = 0;
    for (uint32_t q = tid; q < join_own(a.na_max, lg) / 16; q += JNT)
      reinterpret_cast<uint4*>(cnt_s)[q] = make_uint4(0u, 0u, 0u, 0u);
    sync();
    const uint32_t it = *item0;  // pair index
    if (it == 0xFFFFFFFFu) break;
    if (tid == 0) {
      s_P = a.pairs[it];
      s_kx = s_ky = 0u;
    }
    __syncthreads();
    if (!EPI && warp == 0) {
      const uint32_t gs = pair_threshold(a, it, lane);
      if (lane == 0) s_tau = gs;
    }
    if (tid >= 32 && tid < 32 + (int)T) {
      s_A[tid - 32] = jview(a.join, s_P.ajoin, s_P.nA, tid - 32);
      s_B[tid - 32] = jview(a.join, s_P.bjoin, s_P.nB, tid - 32);
    }
    for (uint32_t i = tid; i < nbo; i += JNT) {  // the bucket offsets of both images
      const uint32_t t = i / (nbk + 1), v = i - t * (nbk + 1);
      off_s[i] = __ldg(jview(a.join, s_P.ajoin, s_P.nA, t).off + v);
      off_s[nbo + i] = __ldg(jview(a.join, s_P.bjoin, s_P.nB, t).off + v);
    }
    if constexpr (EPI) {  // (non-negative floats order as integers)
      const float2* kpb = reinterpret_cast<const float2*>(a.kpts) + s_P.b0;
      float mx = 0.f, my = 0.f;
      for (uint32_t j = tid; j < s_P.nB; j += JNT) {
        const float2 pc = __ldg(kpb + j);
        mx = fmaxf(mx, fabsf(pc.x));
        my = fmaxf(my, fabsf(pc.y));
      }
      mx = __uint_as_float(__reduce_max_sync(0xFFFFFFFFu, __float_as_uint(mx)));
      my = __uint_as_float(__reduce_max_sync(0xFFFFFFFFu, __float_as_uint(my)));
      if (lane == 0) {
        atomicMax(&s_kx, __float_as_uint(mx));
        atomicMax(&s_ky, __float_as_uint(my));
      }
    }
    __syncthreads();
    uint32_t h_thr = h_user;
    if (!EPI) {
      const uint32_t ts = s_tau;  // 0: no guess; else threshold + 1
      if (ts != 0 && ts - 1u < h_thr) h_thr = ts - 1u;
    }
    const bool cut = h_thr < h_user;  // the guess may turn candidates away
    const float2* kpa = EPI ? reinterpret_cast<const float2*>(a.kpts) + s_P.a0 : nullptr;
    const BandRows band{lines, lhi, EPI ? a.F + 9 * (size_t)it : nullptr, kpa, dd};
    if constexpr (EPI) {  // the queries' lines, spread over the cluster
      for (uint32_t q = rank * JNT + tid; q < s_P.nA; q += JNT << lg) {
        float4 l;
        float hi;
        band_line(band.F, __ldg(kpa + q), dd, __uint_as_float(s_kx), __uint_as_float(s_ky), l, hi);
        lines[q] = l;
        lhi[q] = hi;
      }
      sync();
    }

    // ---- scan: a table at a time (a query lies in one bucket of it, so its list and counter have one
    // writer), one warp per bucket (or part of its queries, when there are few buckets), one query per lane
    // against the bucket's candidates ----
    for (uint32_t t = 0; t < T; ++t) {
      for (;;) {
        uint32_t v = 0;
        if (lane == 0) v = atomicAdd(task0 + t, 1u);
        v = __shfl_sync(0xFFFFFFFFu, v, 0);
        if (v >= nbk << nsp) break;
        const uint32_t* o = off_s + t * (nbk + 1) + (v >> nsp);
        uint32_t qs = o[0], nq = o[1] - qs;
        const uint32_t cs = o[nbo], nc = o[nbo + 1] - cs;
        if (nsp) {
          const uint32_t part = v & ((1u << nsp) - 1u), n = nq;
          qs += (uint32_t)(((uint64_t)n * part) >> nsp);
          nq = (uint32_t)(((uint64_t)n * (part + 1)) >> nsp) - (uint32_t)(((uint64_t)n * part) >> nsp);
        }
        if (nq == 0) continue;
        for (uint32_t c0 = 0; c0 < nc; c0 += JCOL) {
          const uint32_t nb = min(JCOL, nc - c0);
#pragma unroll
          for (uint32_t u = 0; u < JCOL; u += 32)
            if (u + lane < nb) {
              w.col[u + lane] = __ldg(s_B[t].rec + cs + c0 + u + lane);
              const uint32_t jj = __ldg(s_B[t].idx + cs + c0 + u + lane);
              w.colj[u + lane] = jj;
              if constexpr (EPI) w.colp[u + lane] = __ldg(reinterpret_cast<const float2*>(a.kpts) + s_P.b0 + jj);
            }
          __syncwarp();
          if constexpr (EPI) scan_rows_band(w, s_A[t], qs, nq, nb, h_thr, L, band, lane);
          else scan_rows(w, s_A[t], qs, nq, nb, h_thr, L, lane);
        }
      }
      sync();
    }

    // ---- finalise: top-k of the survivors, distances, ratio test ----
    for (uint32_t k = warp; ((k << lg) + rank) * 32 < s_P.nA; k += JNT / 32) {
      const uint32_t q = ((k << lg) + rank) * 32 + lane;
      finalise_warp<KC, EPI>(a, s_P, it, cut, q, q < s_P.nA, q < s_P.nA ? cnt_s[k * 32 + lane] : 0u,
                               L.seg + (size_t)q * JSEG, key_s + warp * 32 * join_kp(KC),
                               dist_s + warp * 32 * join_kp(KC), s_hist);
    }
    __syncthreads();
    if (!EPI && !a.tau_fixed)
      for (uint32_t b = tid; b < HBINS; b += JNT)
        if (s_hist[b]) atomicAdd(a.jhist + (size_t)it * HBINS + b, s_hist[b]);
  }
  if constexpr (CL) cl.sync();  // (no CTA leaves while another may read its shared memory)
}

// Threshold guess for pairs that have none yet, from CAL_SAMPLES sampled
// queries (one CTA per pair, one thread per query): the exact k-th Hamming
// distance of each, then the second largest of them plus CAL_MARGIN.  Only a
// performance hint; results never depend on it.
template <int KC>
__global__ void __launch_bounds__(CAL_SAMPLES) k_join_calibrate(MatchArgs a) {
  __shared__ uint32_t s_top[CAL_SAMPLES / 32][2];
  const KParams kp = a.kp;
  const uint32_t T = kp.n_tables, K = kp.top_k;
  const uint32_t thr_user = kp.tau < kp.code_bits ? ((kp.tau + 1u) << 24) : KEY_INF;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  for (uint32_t p = blockIdx.x; p < a.n_pairs; p += gridDim.x) {
    if (*reinterpret_cast<volatile uint32_t*>(a.tau_pair + p) != 0) continue;  // uniform over the CTA
    const PairInfo P = a.pairs[p];
    if (P.nA == 0 || P.nB == 0) continue;
    const uint32_t q = (uint32_t)(((uint64_t)threadIdx.x * P.nA) / CAL_SAMPLES);
    const uint4 qc = __ldg(reinterpret_cast<const uint4*>(a.codes) + P.a0 + q);
    const uint2 qb = __ldg(reinterpret_cast<const uint2*>(a.buckets) + P.a0 + q);
    uint32_t top[KC];
#pragma unroll
    for (int s = 0; s < KC; ++s) top[s] = KEY_INF;
    for (uint32_t t = 0; t < T; ++t) {
      const JView B = jview(a.join, P.bjoin, P.nB, t);
      const uint32_t v = (t < 4 ? (qb.x >> (8 * t)) : (qb.y >> (8 * (t - 4)))) & 0xFFu;
      const uint32_t cs = __ldg(B.off + v), ce = __ldg(B.off + v + 1);
      for (uint32_t c = cs; c < ce; ++c) {
        const uint32_t key = (jt_hamming(__ldg(B.rec + c), qc) << 24) | __ldg(B.idx + c);
        if (key >= thr_user) continue;
        if (key < top[KC - 1]) jt_insert<KC>(top, key);
      }
    }
    const uint32_t kth = jt_kth<KC>(top, K);
    const uint32_t hk = kth == KEY_INF ? 0xFFFFFFFFu : (kth >> 24);  // fewer than k candidates: largest
    // the two largest values of the warp, then of the CTA
    uint32_t m1 = hk;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) m1 = max(m1, __shfl_xor_sync(0xFFFFFFFFu, m1, o));
    const uint32_t eq = __ballot_sync(0xFFFFFFFFu, hk == m1);
    uint32_t m2 = (hk == m1 && (eq & ((1u << lane) - 1u)) == 0) ? 0u : hk;  // drop one copy of the maximum
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) m2 = max(m2, __shfl_xor_sync(0xFFFFFFFFu, m2, o));
    if (lane == 0) {
      s_top[warp][0] = m1;
      s_top[warp][1] = m2;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
      uint32_t b1 = 0, b2 = 0;
      for (int w = 0; w < CAL_SAMPLES / 32; ++w)
        for (int k = 0; k < 2; ++k) {
          const uint32_t x = s_top[w][k];
          if (x > b1) {
            b2 = b1;
            b1 = x;
          } else if (x > b2) {
            b2 = x;
          }
        }
      // two or more samples with fewer than k candidates: leave the pair without a guess
      if (b2 != 0xFFFFFFFFu) atomicMax(a.tau_pair + p, b2 + CAL_MARGIN + 1u);
    }
    __syncthreads();
  }
}

// ---------------------------------------------------------------------------
namespace {

using JoinKernel = void (*)(MatchArgs);
template <bool CL, bool EPI>
JoinKernel join_kernel_kc(uint32_t k) {
  return k <= 4    ? k_join<4, CL, EPI>
         : k <= 8  ? k_join<8, CL, EPI>
         : k <= 10 ? k_join<10, CL, EPI>
         : k <= 16 ? k_join<16, CL, EPI>
                   : k_join<32, CL, EPI>;
}
JoinKernel join_kernel(uint32_t k, uint32_t lg, bool epi) {
  if (epi) return lg ? join_kernel_kc<true, true>(k) : join_kernel_kc<false, true>(k);
  return lg ? join_kernel_kc<true, false>(k) : join_kernel_kc<false, false>(k);
}
JoinKernel calibrate_kernel(uint32_t k) {
  return k <= 4    ? k_join_calibrate<4>
         : k <= 8  ? k_join_calibrate<8>
         : k <= 10 ? k_join_calibrate<10>
         : k <= 16 ? k_join_calibrate<16>
                   : k_join_calibrate<32>;
}

// Launch configuration: grid CTAs in clusters of 2^lg.
void join_config(cudaLaunchConfig_t& cfg, cudaLaunchAttribute& at, uint32_t grid, uint32_t lg, size_t smem,
                 cudaStream_t s) {
  at.id = cudaLaunchAttributeClusterDimension;
  at.val.clusterDim.x = 1u << lg;
  at.val.clusterDim.y = at.val.clusterDim.z = 1;
  cfg.gridDim = dim3(grid);
  cfg.blockDim = dim3(JNT);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cfg.attrs = &at;
  cfg.numAttrs = 1;
}

// CTAs (2^lg) that share a pair.  One, when the pairs fill the GPU's resident CTAs (two per SM): the barrier
// between tables costs more the more warps share a pair (4,950 pairs: 16.7 ms with one CTA, 19.5 with four).  With
// fewer pairs a cluster of up to 8 CTAs, as long as all clusters are resident (66 pairs of 1,000 to 5,000
// features: 0.28 ms with one CTA per pair, 0.126 with four).
uint32_t join_lg(uint32_t n_items, int nsm) {
  uint32_t lg = 0;
  while (lg < 3 && ((uint64_t)n_items << (lg + 1)) <= 2ull * (uint64_t)nsm) ++lg;
  return lg;
}

}  // namespace

uint32_t join_grid(const KParams& kp, uint32_t na_max, uint32_t n_items, uint32_t ctas_per_sm) {
  const bool epi = kp.epi_px >= 0.0;
  // The largest query image: what 32-bit counters of a CTA of JT threads leave room for (k_join_tc's limit, and what
  // the plans' kernel rules were measured with); above it the per-query kernel.  Counters of a byte would let this
  // kernel take more; larger images were not measured with it.
  if ((size_t)4 * ((na_max + 3) / 4 * 4) + (size_t)2 * join_kc(kp.top_k) * JT * 4 + 4096 > 227u * 1024u) return 0;
  int dev = 0, nsm = 0, ncl = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
  const uint32_t lg = join_lg(n_items, nsm);
  const size_t smem = join_smem_bytes(join_kc(kp.top_k), kp.n_tables, na_max, lg, epi);
  const JoinKernel kern = join_kernel(kp.top_k, lg, epi);
  const uint32_t ctas = join_resident(kern, smem, lg ? 1u : n_items, ctas_per_sm, JNT);
  if (!lg || !ctas) return ctas;
  cudaLaunchConfig_t cfg{};
  cudaLaunchAttribute at{};
  join_config(cfg, at, 1u << lg, lg, smem, 0);
  if (cudaOccupancyMaxActiveClusters(&ncl, kern, &cfg) != cudaSuccess || ncl < 1) {
    cudaGetLastError();
    return 0;
  }
  if (ctas_per_sm && (ncl << lg) > nsm * (int)ctas_per_sm) ncl = (nsm * (int)ctas_per_sm) >> lg;
  return n_items < (uint32_t)ncl ? n_items : (uint32_t)(ncl > 0 ? ncl : 1);
}

cudaError_t launch_join_calibrate(const MatchArgs& a, cudaStream_t s) {
  if (a.n_pairs == 0 || a.kp.epi_px >= 0.0) return cudaSuccess;  // the band form uses no threshold guess
  int dev = 0, nsm = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
  const uint32_t grid = a.n_pairs < (uint32_t)nsm * 8 ? a.n_pairs : (uint32_t)nsm * 8;
  calibrate_kernel(a.kp.top_k)<<<grid, CAL_SAMPLES, 0, s>>>(a);
  return cudaGetLastError();
}

cudaError_t launch_join(const MatchArgs& a, uint32_t grid, cudaStream_t s) {
  if (a.n_items == 0 || grid == 0) return cudaSuccess;
  const bool epi = a.kp.epi_px >= 0.0;
  int dev = 0, nsm = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
  const uint32_t lg = join_lg(a.n_items, nsm);
  const size_t smem = join_smem_bytes(join_kc(a.kp.top_k), a.kp.n_tables, a.na_max, lg, epi);
  if (!lg) {
    join_kernel(a.kp.top_k, 0, epi)<<<grid, JNT, smem, s>>>(a);
    return cudaGetLastError();
  }
  cudaLaunchConfig_t cfg{};
  cudaLaunchAttribute at{};
  join_config(cfg, at, grid << lg, lg, smem, s);
  return cudaLaunchKernelEx(&cfg, join_kernel(a.kp.top_k, lg, epi), a);
}

}  // namespace chx
