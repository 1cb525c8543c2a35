// Lookup tables of Step 1 (Sec. 3.1): for each candidate image, each table t
// and each m-bit short code v, the list of points whose code in table t is v.
//
// Layout (private to the library): each image's features are cut into chunks
// of JC features; chunk k (numbered over the whole set) occupies
// chunk_bytes(T) bytes at tables + k * chunk_bytes(T):
//   uint16 off[T][OFF_STRIDE]  bucket v of table t holds local indices
//                              idx[t][off[t][v] .. off[t][v+1])
//   uint16 idx[T][JC]          local feature indices (0..JC-1), ascending
//                              within a bucket (stable counting sort)
// A chunk is staged whole into shared memory by the matcher.
#include "internal.h"

namespace chx {

// Stable counting sort of one (image or chunk, table) in shared memory, one
// CTA of NW warps, for at most BJ_MAX_N features.  Warp w takes the w-th NW-th
// of the features; its bucket cursors start after the earlier warps' entries
// of the same bucket, so the order within a bucket is the feature order.  The
// sorted local indices are then written out in order (and, for the join
// tables, the codes gathered behind them), so every global write is
// coalesced.
//   blockIdx.x < join_tasks: the join tables of image blockIdx.x / T (the
//                  join_block layout: uint32 offsets, uint32 indices, inline codes);
//   else:          lookup-table chunk (blockIdx.x - join_tasks) / T of the layout above.
// The rank among a warp's 32 features comes from 8 ballots, one per bucket bit:
// match.any takes its time per distinct value, and nearly all 32 are.  A build of
// 773,191 features: 338 us with match.any and two launches, 313 with ballots, 297
// in one launch; 321,454: 176, 159, 151; 4,000: 40.4, 39.6, 35.1.  What is left waits
// for the gathered codes and for shared memory.
constexpr uint32_t BJ_MAX_N = 65535;  // local indices held as uint16 in shared memory

template <int NW>
__global__ void __launch_bounds__(NW * 32) k_sort_tables(const uint8_t* __restrict__ buckets,
                                                         const uint32_t* __restrict__ codes,
                                                         const uint64_t* __restrict__ img_f0,
                                                         const uint32_t* __restrict__ img_n,
                                                         const uint64_t* __restrict__ img_join,
                                                         const uint64_t* __restrict__ chunk_f0,
                                                         const uint32_t* __restrict__ chunk_len, uint32_t T,
                                                         uint32_t join_tasks, uint8_t* __restrict__ out) {
  extern __shared__ __align__(16) uint32_t bsm[];
  constexpr uint32_t NT = NW * 32;
  uint32_t* hist = bsm;  // [NW warps][256 buckets]
  __shared__ uint32_t s_wsum[8];
  const uint32_t tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
  const bool chunk = blockIdx.x >= join_tasks;
  const uint32_t task = blockIdx.x - (chunk ? join_tasks : 0u), u = task / T, t = task % T;
  const uint64_t f0 = chunk ? chunk_f0[u] : img_f0[u];
  const uint32_t n = chunk ? chunk_len[u] : img_n[u];
  uint16_t* sidx = reinterpret_cast<uint16_t*>(bsm + NW * 256);      // [n] sorted local indices
  uint8_t* sb = reinterpret_cast<uint8_t*>(sidx + (n + 7) / 8 * 8);  // [n] bucket of each feature
  for (uint32_t k = tid; k < NW * 256; k += NT) hist[k] = 0;
  const uint8_t* bsrc = buckets + f0 * 8 + t;
#pragma unroll 8
  for (uint32_t j = tid; j < n; j += NT) sb[j] = __ldg(bsrc + (uint64_t)j * 8);
  __syncthreads();
  const uint32_t seg = (n + NW - 1) / NW, j_lo = min(n, w * seg), j_hi = min(n, j_lo + seg);
  uint32_t* hw = hist + w * 256;
  for (uint32_t j = j_lo + lane; j < j_hi; j += 32) atomicAdd(&hw[sb[j]], 1u);
  __syncthreads();
  // thread b < 256: bucket b's total, its exclusive offset over buckets, and the
  // warps' starting cursors in bucket b
  const uint32_t b = tid;
  uint32_t tot = 0, incl = 0;
  if (b < 256) {
#pragma unroll
    for (int k = 0; k < NW; ++k) tot += hist[k * 256 + b];
    incl = tot;
#pragma unroll
    for (uint32_t d = 1; d < 32; d <<= 1) {
      const uint32_t o = __shfl_up_sync(0xFFFFFFFFu, incl, d);
      if (lane >= d) incl += o;
    }
    if (lane == 31) s_wsum[w] = incl;
  }
  __syncthreads();
  uint32_t excl = incl - tot;
  if (b < 256)
    for (uint32_t k = 0; k < w; ++k) excl += s_wsum[k];
  uint8_t* blk;
  if (chunk) {
    blk = out + (uint64_t)u * chunk_bytes(T);
    uint16_t* off = reinterpret_cast<uint16_t*>(blk) + (size_t)t * OFF_STRIDE;
    if (b < 256) off[b] = (uint16_t)excl;
    if (b == 255) off[256] = (uint16_t)(excl + tot);
  } else {
    blk = out + img_join[u] + (uint64_t)t * join_block(n);
    uint32_t* off = reinterpret_cast<uint32_t*>(blk);
    if (b < 256) off[b] = excl;
    if (b == 255) off[256] = excl + tot;
  }
  if (b < 256) {
    uint32_t run = excl;
#pragma unroll
    for (int k = 0; k < NW; ++k) {
      const uint32_t c = hist[k * 256 + b];
      hist[k * 256 + b] = run;
      run += c;
    }
  }
  __syncthreads();
  // stable scatter of each warp's range, 32 features at a time in feature order
  const uint32_t lt = (1u << lane) - 1u;
  for (uint32_t j0 = j_lo; j0 < j_hi; j0 += 32) {
    const uint32_t j = j0 + lane;
    const bool valid = j < j_hi;
    const uint32_t bk = valid ? (uint32_t)sb[j] : 0u;
    uint32_t peers = __ballot_sync(0xFFFFFFFFu, valid);  // valid lanes of the same bucket
#pragma unroll
    for (uint32_t i = 0; i < 8; ++i) {
      const uint32_t one = __ballot_sync(0xFFFFFFFFu, bk >> i & 1u);
      peers &= bk >> i & 1u ? one : ~one;
    }
    const uint32_t rank = __popc(peers & lt);
    uint32_t pos = 0;
    if (valid) pos = hw[bk] + rank;
    __syncwarp();
    if (valid) {
      sidx[pos] = (uint16_t)j;
      if (rank == 0) hw[bk] += __popc(peers);
    }
    __syncwarp();
  }
  __syncthreads();
  if (chunk) {
    uint16_t* idx = reinterpret_cast<uint16_t*>(blk) + (size_t)T * OFF_STRIDE + (size_t)t * JC;
    for (uint32_t p = tid; p < n; p += NT) idx[p] = sidx[p];
  } else {
    uint32_t* idx = reinterpret_cast<uint32_t*>(blk + 1040);
    uint4* rec = reinterpret_cast<uint4*>(blk + 1040 + 4 * ((n + 3) / 4 * 4));
    const uint4* cd = reinterpret_cast<const uint4*>(codes) + f0;
#pragma unroll 4
    for (uint32_t p = tid; p < n; p += NT) {
      const uint32_t j = sidx[p];
      idx[p] = j;
      rec[p] = __ldg(cd + j);
    }
  }
}

// Warps of a CTA: 8 where images are small and their CTAs more than the SMs, else 16.  A CTA clears and adds up a
// histogram per warp whatever it sorts, and twice the CTAs fit an SM; few CTAs, and large images, gain from the
// warps.  us a build with 8 / 16 (6 tables): 2,000 images of 64 features 138 / 209, 256 234 / 308, 1,000 of 1,000 341 /
// 373, 200 of 4,000 276 / 282, 100 of 8,000 288 / 281, 2 of 1,000 39.6 / 37.3, 2 of 4,000 45.4 / 43.6.
int tables_warps(uint32_t n_max, uint64_t tasks, int nsm) { return n_max <= 4096 && tasks > (uint64_t)nsm ? 8 : 16; }

static size_t sort_smem(uint32_t n_max, int nw) { return nw * 256 * 4 + (size_t)(n_max + 7) / 8 * 8 * 3; }

// Join tables of a set with an image of more than BJ_MAX_N features: one warp
// per (image, table), a stable counting sort over the whole image with global
// scatters.
__global__ void __launch_bounds__(256) k_build_join(const uint8_t* __restrict__ buckets,
                                                    const uint32_t* __restrict__ codes,
                                                    const uint64_t* __restrict__ img_f0,
                                                    const uint32_t* __restrict__ img_n,
                                                    const uint64_t* __restrict__ img_join, uint32_t n_images,
                                                    uint32_t T, uint8_t* __restrict__ join) {
  __shared__ uint32_t cur_all[8][256];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const uint64_t task = (uint64_t)blockIdx.x * 8 + w;
  if (task >= (uint64_t)n_images * T) return;  // whole warp leaves together
  const uint32_t im = (uint32_t)(task / T), t = (uint32_t)(task % T);
  const uint64_t f0 = img_f0[im];
  const uint32_t n = img_n[im];
  uint8_t* blk = join + img_join[im] + (uint64_t)t * join_block(n);
  uint32_t* off = reinterpret_cast<uint32_t*>(blk);
  uint32_t* idx = reinterpret_cast<uint32_t*>(blk + 1040);
  uint4* rec = reinterpret_cast<uint4*>(blk + 1040 + 4 * ((n + 3) / 4 * 4));
  uint32_t* cur = cur_all[w];
#pragma unroll
  for (int k = 0; k < 8; ++k) cur[lane * 8 + k] = 0;
  __syncwarp();
  for (uint32_t j = lane; j < n; j += 32) atomicAdd(&cur[buckets[(f0 + j) * 8 + t]], 1u);
  __syncwarp();
  uint32_t v[8], run = 0;
#pragma unroll
  for (int k = 0; k < 8; ++k) {
    v[k] = run;
    run += cur[lane * 8 + k];
  }
  uint32_t incl = run;
#pragma unroll
  for (int d = 1; d < 32; d <<= 1) {
    const uint32_t o = __shfl_up_sync(0xFFFFFFFFu, incl, d);
    if (lane >= d) incl += o;
  }
  const uint32_t excl = incl - run;
  __syncwarp();
#pragma unroll
  for (int k = 0; k < 8; ++k) {
    off[lane * 8 + k] = excl + v[k];
    cur[lane * 8 + k] = excl + v[k];
  }
  if (lane == 31) off[256] = incl;
  __syncwarp();
  const uint32_t lt = (1u << lane) - 1u;
  const uint4* cd = reinterpret_cast<const uint4*>(codes) + f0;
  for (uint32_t j0 = 0; j0 < n; j0 += 32) {
    const uint32_t j = j0 + lane;
    const bool valid = j < n;
    const uint32_t b = valid ? (uint32_t)buckets[(f0 + j) * 8 + t] : 256u + lane;
    const uint32_t peers = __match_any_sync(0xFFFFFFFFu, b);
    const uint32_t rank = __popc(peers & lt);
    uint32_t pos = 0;
    if (valid) pos = cur[b] + rank;
    __syncwarp();
    if (valid) {
      idx[pos] = j;
      rec[pos] = __ldg(cd + j);
      if (rank == 0) cur[b] += __popc(peers);
    }
    __syncwarp();
  }
}

// Image and chunk tables in one launch while the images' shared memory leaves room for four CTAs of an SM, as many
// as its threads do (up to 13,640 features); else the chunks would run fewer at a time than they can.  An SM has 228
// KB, of which the system takes 1 KB for each CTA and the kernel's static arrays 32 bytes.
bool tables_one_launch(uint32_t n_max) { return sort_smem(n_max, 16) <= 228 * 1024 / 4 - 1024 - 32; }

cudaError_t launch_build_tables(const uint8_t* buckets, const uint32_t* codes, const uint64_t* img_f0,
                                const uint32_t* img_n, const uint64_t* img_join, uint32_t n_images, uint32_t n_max,
                                const uint64_t* chunk_f0, const uint32_t* chunk_len, uint32_t n_chunks,
                                uint32_t n_tables, uint8_t* tables, cudaStream_t s) {
  const uint64_t jt = (uint64_t)n_images * n_tables, ct = (uint64_t)n_chunks * n_tables;
  if (jt > 0x7FFFFFFFull || ct > 0x7FFFFFFFull || jt + ct > 0x7FFFFFFFull)
    return cudaErrorInvalidValue;  // one CTA (or warp) per image or chunk and table
  static_assert(JC <= (int)BJ_MAX_N, "chunk tables sort in shared memory");
  static int attr_dev = -1;
  int dev = 0, nsm = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (attr_dev != dev) {  // (8 warps: at most 20 KB)
    e = cudaFuncSetAttribute(k_sort_tables<16>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)sort_smem(BJ_MAX_N, 16));
    if (e != cudaSuccess) return e;
    attr_dev = dev;
  }
  cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
  auto sort = [&](uint64_t join_tasks, uint64_t tasks, uint32_t n) {
    if (tasks == 0) return cudaSuccess;
    const int nw = tables_warps(n_max, tasks, nsm);
    (nw == 8 ? k_sort_tables<8> : k_sort_tables<16>)<<<(unsigned)tasks, nw * 32, sort_smem(n, nw), s>>>(
        buckets, codes, img_f0, img_n, img_join, chunk_f0, chunk_len, n_tables, (uint32_t)join_tasks, tables);
    return cudaGetLastError();
  };
  if (tables_one_launch(n_max)) return sort(jt, jt + ct, n_max);
  e = sort(0, ct, JC);
  if (e != cudaSuccess || jt == 0) return e;
  if (n_max <= BJ_MAX_N) return sort(jt, jt, n_max);
  k_build_join<<<(unsigned)((jt + 7) / 8), 256, 0, s>>>(buckets, codes, img_f0, img_n, img_join, n_images, n_tables,
                                                        tables);
  return cudaGetLastError();
}

}  // namespace chx
