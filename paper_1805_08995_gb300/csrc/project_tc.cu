// Projection of Sec. 5.1 on tcgen05 tensor cores (sm_103a), for either precision setting.
//
// v_fb = sum_j R_bj x_fj - c_b.  Row b of R is scaled by 2^s_b so that its largest entry lies in (256, 512] (a row
// of zeros or of numbers below 2^-990 may stay smaller) and split into three f16 terms:
//   r = 2^s R_bj,  hi = rint(r),  mid = rint(2^11 (r - hi)),  lo = 2^-11 rint(2^22 (r - hi) - 2^11 mid),
// integers (lo: multiples of 2^-11) of up to 10 bits and the sign each, so normal f16 numbers.
// x, 0 .. 255, is exact in f16.  One accumulator takes X hi^T: integers of at most 128 * 255 * 512 < 2^24, exact in
// FP32 in any order.  A second one takes X mid^T, then X lo^T, and enters at 2^-11.  Error of A + 2^-11 B - c
// against 2^s v, in units of N = max(2^s ||R_b||, 256) ||x||:
//   * the split: |r - hi - 2^-11 (mid + lo)| <= 2^-23, so at most 2^-23 sum x <= 2^-23 sqrt(128) ||x|| < 2^-27 N;
//   * B, 16 MMAs of 16 products.  How the tensor cores add is not documented; taken here: each MMA aligns its products
//     and the accumulator to the largest of them and cuts all off below its 24th bit, and the sum as well (A stays
//     exact under that: integers).  288 cuts of at most 2^-23 S each, S = sum x (|mid| + |lo|) <= 1024.5 sqrt(128)
//     ||x||, at 2^-11: below 2^-20.3 N for a row with one large entry (N = 256 ||x||; for rows of normal numbers, N =
//     1900 ||x||, seven times less);
//   * A + 2^-11 B rounded: 2^-24 N; minus c: 2^-24 (N + |c|), and c is rounded itself: beta has 2^-23 |c|.
// The sum is below 2^-20.1 N; the flag test takes 2^-20 N plus beta (which has the rounding of the double sequence
// too).  |v~| under the bound goes to k_fix_fp64, so the signs equal the double definition.
//
// Before, the FP32 setting took CUDA-core FMA chains over 24-bit weights (bound 2^-16) and the other one a two-term
// bf16 split (2^-15).  Against the doubles, over 60,000 features and 176 rows of normal numbers: error 1.9e-5 rms and
// 1.7e-4 at most, where the FMA chains had 1.1e-4 and 1.5e-3 and the bf16 split 1.3e-3 and 6.6e-3; of 844,018
// features 2,169 projections are re-evaluated, where it was 34,262 and 68,755 (1,063 with half the bound, which a row of
// one large entry could exceed; 773,191 features 2 us a build).
//
// Shared-memory operands use the canonical K-major layout without swizzle: 8-row x 16-byte core matrices of 128
// contiguous bytes; core matrix (r8, k8) sits at (r8 * 16 + k8) * 128 bytes, so the leading-dimension offset (next
// core matrix along K) is 128 B and the stride offset (next 8 rows) is 2 KB.
//
// One CTA per SM, persistent over tiles of 128 features, two operand buffers.  The rows of R are taken in two halves
// of up to 96 (one if all fit), each with its own two accumulators and mbarrier: while 16 warps read one half back
// (feature row r is TMEM lane r; the four warps that may access a lane take 24 rows each), the tensor cores work on
// the other.  hi and mid are multiplied side by side (N = 192), which reads the features from shared memory once for
// both.  A 17th warp issues the MMAs, so the others only announce that they have read a half (an arrival on the half's
// second mbarrier) and go on.
// 773,191 features, 176 rows: 139 us (with all warps at a barrier per half and N = 96: 159; bf16 form 190); 321,454:
// 63 us (73; FP32 form 450).  Bound by issue and the latency of the read-back (issue 46 %, tensor pipe 32 % active).
//
// Every wait between the first tile and the last is a bounded one on an mbarrier: for a half's MMAs, for all warps to
// have read a half, for the signs of a tile.  A warp whose wait times out records an error and leaves its loop; those
// that depend on it leave at a time-out of their own.  The issuing warp then waits (bounded) for what is in flight, all
// warps meet at the last barrier, and the tensor memory is released.
#include "tc_common.cuh"

namespace chx {

constexpr int TC_M = 128;
constexpr int TC_K = 128;
constexpr int TC_NH = 96;                // rows of R per half
constexpr uint32_t TC_TMEM_COLS = 512;   // 2 halves x 2 accumulators x 96 columns
constexpr int PT_WORK = 512;              // 16 warps convert, read back and write
constexpr int PT_THREADS = PT_WORK + 32;  // and one issues the MMAs

// One arrival on an mbarrier for the whole warp, after what its lanes have read and written.
__device__ __forceinline__ void warp_arrive(uint32_t mbar, int lane) {
  __syncwarp();
  if (lane == 0) asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(mbar) : "memory");
}

// Two bytes of w (half 0: bytes 0, 1; half 1: bytes 2, 3) as f16x2, exact: 0x64bb is 1024 + bb.
__device__ __forceinline__ uint32_t f16x2_of_bytes(uint32_t w, int half) {
  const uint32_t x = __byte_perm(w, 0x64646464u, half ? 0x4342 : 0x4140);
  uint32_t r;
  asm("sub.rn.f16x2 %0, %1, %2;" : "=r"(r) : "r"(x), "r"(0x64006400u));
  return r;
}

// 8 consecutive accumulator columns of this thread's TMEM lane (no wait).
__device__ __forceinline__ void tmem_ld8_nowait(uint32_t taddr, uint32_t (&r)[8]) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
               : "r"(taddr));
}

template <bool DBG>
__global__ void __launch_bounds__(PT_THREADS, 1) k_project(const uint8_t* __restrict__ desc, uint64_t n,
                                                           const uint4* __restrict__ Rs, uint32_t NP,
                                                           const RowConst* __restrict__ rcg, KParams kp,
                                                           uint32_t* __restrict__ codes,
                                                           uint8_t* __restrict__ buckets,
                                                           uint32_t* __restrict__ sqnorm,
                                                           uint32_t* __restrict__ flagmask,
                                                           uint32_t* __restrict__ flaglist,
                                                           unsigned long long* __restrict__ nflag_feat,
                                                           uint32_t* __restrict__ status,
                                                           float* __restrict__ dbg_x, float* __restrict__ dbg_e) {
  extern __shared__ __align__(128) uint8_t tsm[];
  __shared__ __align__(8) uint64_t s_mbar[2];  // per half: its MMAs are done
  __shared__ __align__(8) uint64_t s_read[2];  // per half: every warp has read it (and written the next tile's operand)
  __shared__ uint32_t s_tmem;
  __shared__ float4 rc[PT_ROWS_TC];            // c, alpha, beta
  __shared__ float s_nx[3][TC_M];              // [tile % 3][row]: ||x||
  __shared__ uint32_t s_bits[2][8][TC_M];      // [tile parity][24 rows of R][row]: signs
  __shared__ uint32_t s_flag[2][6][TC_M];      // [tile parity][word][row]: rows under the bound (zero in between)
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int cg = warp >> 2;                                       // 24 of a half's 96 rows of R
  const uint32_t r = (uint32_t)((warp & 3) * 32 + lane);          // feature row in the tile = TMEM lane
  uint8_t* As = tsm;                                              // 2 x 32 KB
  uint8_t* Bs = tsm + 2 * (TC_M * TC_K * 2);                      // per half its rows of hi, mid and lo, 256 B each
  const int halves = NP > TC_NH ? 2 : 1;

  for (uint32_t i = tid; i < NP * (3 * TC_K * 2 / 16); i += PT_THREADS) reinterpret_cast<uint4*>(Bs)[i] = __ldg(Rs + i);
  for (int i = tid; i < PT_ROWS_TC; i += PT_THREADS) {
    RowConst z{};
    if ((uint32_t)i < kp.rows) z = rcg[i];
    rc[i] = make_float4(z.c32, z.alpha, z.beta, 0.f);
  }
  for (int i = tid; i < 2 * 6 * TC_M; i += PT_THREADS) (&s_flag[0][0][0])[i] = 0u;
  if (tid == 0) {
    for (int h = 0; h < 2; ++h) {
      asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(&s_mbar[h])) : "memory");
      asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(&s_read[h])), "n"(PT_WORK / 32) : "memory");
    }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&s_tmem)),
                 "r"(TC_TMEM_COLS)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }

  // 8 features x 4 quarter rows of 32 bytes per warp: conflict-free stores, whole descriptors per warp
  const uint32_t lrow = (uint32_t)(warp * 8 + (lane & 7)), part = (uint32_t)lane >> 3;
  const uint64_t ntiles = (n + TC_M - 1) / TC_M;
  uint4 v[2];
  auto load_tile = [&](uint64_t t) {
    v[0] = v[1] = make_uint4(0u, 0u, 0u, 0u);
    const uint64_t f = t * TC_M + lrow;
    if (t < ntiles && f < n) {
      const uint4* src = reinterpret_cast<const uint4*>(desc + f * DIM) + 2 * part;
      v[0] = __ldg(src);
      v[1] = __ldg(src + 1);
    }
  };
  // the loaded bytes -> f16 operand rows, the norms; sqnorm is written here
  auto convert = [&](uint64_t t, uint32_t k) {  // t: the CTA's k-th tile
    const uint32_t b = k & 1u;
    uint8_t* dst = As + b * (TC_M * TC_K * 2) + (lrow >> 3) * 2048 + (4 * part) * 128 + (lrow & 7) * 16;
    uint32_t sq = 0;
#pragma unroll
    for (int c = 0; c < 2; ++c) {
      const uint32_t w[4] = {v[c].x, v[c].y, v[c].z, v[c].w};
#pragma unroll
      for (int k = 0; k < 4; ++k) sq = __dp4a(w[k], w[k], sq);
#pragma unroll
      for (int k = 0; k < 2; ++k)
        *reinterpret_cast<uint4*>(dst + (2 * c + k) * 128) =
            make_uint4(f16x2_of_bytes(w[2 * k], 0), f16x2_of_bytes(w[2 * k], 1), f16x2_of_bytes(w[2 * k + 1], 0),
                       f16x2_of_bytes(w[2 * k + 1], 1));
    }
    sq += __shfl_xor_sync(0xFFFFFFFFu, sq, 8);
    sq += __shfl_xor_sync(0xFFFFFFFFu, sq, 16);
    if (part == 0) {
      s_nx[k % 3u][lrow] = __fsqrt_ru((float)sq);
      if (t * TC_M + lrow < n) sqnorm[t * TC_M + lrow] = sq;
    }
  };
  // the MMAs of half h of the tile in buffer b (one thread): hi and mid side by side, then lo onto mid's columns
  auto issue = [&](int h, uint32_t b) {
    const uint32_t rows = h ? NP - TC_NH : min(NP, (uint32_t)TC_NH);
    const uint32_t a0 = smem_u32(As) + b * (TC_M * TC_K * 2), b0 = smem_u32(Bs) + (uint32_t)h * (3 * TC_NH * TC_K * 2);
    const uint32_t acc = s_tmem + (uint32_t)h * (2 * TC_NH);
#pragma unroll
    for (int kk = 0; kk < TC_K / 16; ++kk)
      tc_mma(acc, tc_desc(a0 + kk * 256, 128, 2048), tc_desc(b0 + kk * 256, 128, 2048), tc_idesc_f16(TC_M, 2 * rows),
             kk ? 1u : 0u);
#pragma unroll
    for (int kk = 0; kk < TC_K / 16; ++kk)
      tc_mma(acc + rows, tc_desc(a0 + kk * 256, 128, 2048), tc_desc(b0 + rows * (2 * TC_K * 2) + kk * 256, 128, 2048),
             tc_idesc_f16(TC_M, rows), 1u);
    tc_commit(smem_u32(&s_mbar[h]));
  };
  // the whole warp waits for a phase; false: the wait timed out
  auto wait_all = [&](uint64_t* mbar, uint32_t parity) {
    const bool ok = __all_sync(0xFFFFFFFFu, mbar_wait(smem_u32(mbar), parity));
    if (!ok && lane == 0) atomicOr(status, DST_INDEX);  // never expected
    return ok;
  };

  uint64_t tile = blockIdx.x;
  if (tid < PT_WORK) {
    load_tile(tile);
    convert(tile, 0);
    load_tile(tile + gridDim.x);
  }
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  if (tid >= PT_WORK) {  // the issuing warp: a half's next MMAs once all have read its accumulators
    uint32_t last = 0;  // bit h: parity of the phase that half h's latest MMAs complete
    if (lane == 0)
      for (int h = 0; h < halves; ++h) issue(h, 0);
    bool ok = true;
    for (uint32_t k = 0; ok && tile + gridDim.x < ntiles; tile += gridDim.x, ++k) {
      for (int h = 0; h < halves; ++h) {
        ok = wait_all(&s_read[h], k & 1u);
        if (!ok) break;
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        if (lane == 0) issue(h, (k + 1) & 1u);
        last ^= 1u << h;
      }
    }
    // whatever ended the loop: no operand, accumulator or mbarrier goes before the last MMAs are done
    for (int h = 0; h < halves; ++h) wait_all(&s_mbar[h], last >> h & 1u);
  } else {
    const uint32_t lane_base = s_tmem + ((uint32_t)((warp & 3) * 32) << 16);
    bool ok = true;
    for (uint32_t k = 0; ok && tile < ntiles; tile += gridDim.x, ++k) {
      const uint32_t b = k & 1u;
      const uint64_t f = tile * TC_M + r, next = tile + gridDim.x;
      if (next < ntiles) {  // (this thread waited for all MMAs of that buffer in the previous round)
        convert(next, k + 1);
        load_tile(next + gridDim.x);
      }
      float nx = 0.f;
      for (int h = 0; h < halves; ++h) {
        ok = wait_all(&s_mbar[h], b);
        if (!ok) break;
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        if (h == 0) nx = s_nx[k % 3u][r];  // (written before the barrier that this half's MMAs waited for)
        const uint32_t col = lane_base + (uint32_t)(h * 2 * TC_NH + cg * 24);
        const uint32_t rows = h ? NP - TC_NH : min(NP, (uint32_t)TC_NH);
        uint32_t hi[3][8], lo[3][8], pos = 0, out = 0;  // bit 23 - i: row i's sign, and whether it is outside the bound
#pragma unroll
        for (int u = 0; u < 3; ++u) {
          tmem_ld8_nowait(col + u * 8, hi[u]);
          tmem_ld8_nowait(col + rows + u * 8, lo[u]);
        }
        tmem_wait_ld();
        const float4* rh = rc + h * TC_NH + cg * 24;
#pragma unroll
        for (int i = 0; i < 24; ++i) {
          const float4 c = rh[i];
          const float x = fmaf(__uint_as_float(lo[i >> 3][i & 7]), 0x1p-11f, __uint_as_float(hi[i >> 3][i & 7])) - c.x;
          const float E = __fmaf_ru(c.y, nx, c.z);
          if (DBG && f < n && (uint32_t)(h * TC_NH + cg * 24 + i) < kp.rows) {
            const uint64_t o = f * kp.rows + h * TC_NH + cg * 24 + i;
            const int s = -__float_as_int(rcg[h * TC_NH + cg * 24 + i].pad);
            dbg_x[o] = ldexpf(x, s);
            dbg_e[o] = ldexpf(E, s);
          }
          pos = __funnelshift_l(__float_as_uint(x), pos, 1);  // (x = 0 is under the bound)
          out = __funnelshift_l(__float_as_uint(E - fabsf(x)), out, 1);
        }
        // rows under the bound, and beyond the last row nothing
        const int left = (int)kp.rows - (h * TC_NH + cg * 24);
        const uint32_t live = left >= 24 ? 0xFFFFFFu : left <= 0 ? 0u : (1u << left) - 1u;
        const uint32_t fl = (__brev(~out) >> 8) & live;
        s_bits[b][4 * h + cg][r] = (__brev(~pos) >> 8) & live & ~fl;
        if (fl) {  // (rare)
          const int at = h * TC_NH + cg * 24;
          atomicOr(&s_flag[b][at >> 5][r], fl << (at & 31));
          if ((at & 31) > 8) atomicOr(&s_flag[b][(at >> 5) + 1][r], fl >> (32 - (at & 31)));
        }
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
        warp_arrive(smem_u32(&s_read[h]), lane);
      }
      if (!ok) break;
      if (cg == 0 && !wait_all(&s_read[halves - 1], b)) break;  // the warps that write wait for all signs of the tile
      // (the words of a parity are written again only after MMAs that wait for these warps' next arrival)
      if (cg == 0 && f < n) {
        uint32_t w[6], fl[6];
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          uint32_t a[4];
#pragma unroll
          for (int i = 0; i < 4; ++i) a[i] = h < halves ? s_bits[b][4 * h + i][r] : 0u;
          w[3 * h] = a[0] | a[1] << 24;
          w[3 * h + 1] = a[1] >> 8 | a[2] << 16;
          w[3 * h + 2] = a[2] >> 16 | a[3] << 8;
        }
#pragma unroll
        for (int i = 0; i < 6; ++i) {
          fl[i] = s_flag[b][i][r];
          if (fl[i]) s_flag[b][i][r] = 0u;
        }
        write_feature(f, w, fl, kp, codes, buckets, flagmask, flaglist, nflag_feat);
      }
    }
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  if (warp == 0)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(s_tmem), "r"(TC_TMEM_COLS) : "memory");
}

cudaError_t launch_project(const uint8_t* desc, uint64_t n, const void* Rs, uint32_t NP, const RowConst* rc,
                           const KParams& kp, uint32_t* codes, uint8_t* buckets, uint32_t* sqnorm, uint32_t* flagmask,
                           uint32_t* flaglist, unsigned long long* nflag_feat, uint32_t* status, cudaStream_t s,
                           float* dbg_x, float* dbg_e) {
  if (n == 0) return cudaSuccess;
  if (NP % 16 || NP < 16 || NP > PT_ROWS_TC) return cudaErrorInvalidValue;
  const size_t smem = 2 * (size_t)TC_M * TC_K * 2 + 3 * (size_t)NP * TC_K * 2;
  static int attr_dev = -1;
  int dev = 0, nsm = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (attr_dev != dev) {
    const int most = 2 * TC_M * TC_K * 2 + 3 * PT_ROWS_TC * TC_K * 2;
    e = cudaFuncSetAttribute(k_project<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, most);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(k_project<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, most);
    if (e != cudaSuccess) return e;
    attr_dev = dev;
  }
  cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
  const uint64_t ntiles = (n + TC_M - 1) / TC_M;
  const int grid = (int)(ntiles < (uint64_t)nsm ? ntiles : (uint64_t)nsm);
  const uint4* R4 = reinterpret_cast<const uint4*>(Rs);
  if (dbg_x)
    k_project<true><<<grid, PT_THREADS, smem, s>>>(desc, n, R4, NP, rc, kp, codes, buckets, sqnorm, flagmask, flaglist,
                                                   nflag_feat, status, dbg_x, dbg_e);
  else
    k_project<false><<<grid, PT_THREADS, smem, s>>>(desc, n, R4, NP, rc, kp, codes, buckets, sqnorm, flagmask,
                                                    flaglist, nflag_feat, status, dbg_x, dbg_e);
  return cudaGetLastError();
}

}  // namespace chx
