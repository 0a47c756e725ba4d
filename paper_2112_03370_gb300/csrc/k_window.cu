// Pixel windows of time-aligned detector groups: the un-pointing P and pointing P^T of the FP32
// A-application (Sect. 3.1, MAPMAT and the local pixel indexation).
//
// Detectors of one focal plane observe nearly the same sky at the same time, so the samples of a
// group of detectors over a short window of time fall on few distinct pixels (ground raster, all
// detectors x 64 samples: 9.6 samples per pixel; satellite spin scan: 3.4), while one detector's
// own samples almost never repeat a pixel within a tile.  The plan gives each sample the rank of
// its pixel among the sorted distinct pixels of its group (a uint16 slot), so
//   P:   a CTA loads the group's map entries once into shared memory and every sample reads its
//        (I, Q, U) from there;
//   P^T: the group's samples, ordered by slot once at plan time, are summed run by run in registers
//        and each run is added to the global map with one vector atomic (the local reduction before
//        the global one of Sect. 3.1).
// The weights (cos 2psi, sin 2psi) are evaluated in registers from the angle 2psi reduced to
// [-pi, pi] once at plan time in FP64, so the kernels stream 6 bytes of pointing per sample
// (slot + angle) instead of a pixel index and two precomputed weights.
#include <algorithm>

#include "df64.cuh"
#include "mm_internal.cuh"

namespace mm {

namespace {

constexpr int kHashBits = 13;
constexpr int kHash = 1 << kHashBits;   // open-addressing set, twice the window capacity
static_assert(kHash >= 2 * kWinCap, "hash set must be sparse");
constexpr int kWarps = kWinThreads / 32;

__device__ __forceinline__ uint32_t hash_of(int32_t p) {
  return ((uint32_t)p * 2654435761u) >> (32 - kHashBits);   // Knuth's multiplicative hash
}

// The chunk of block b that belongs to a group: samples [lo, lo + len) of the global order.
__device__ __forceinline__ void group_chunk(const PGroup& G, const int64_t* __restrict__ block_off, int c,
                                            int64_t& lo, int& len) {
  const int b = G.b0 + c * G.b_stride;
  const int64_t blo = __ldg(block_off + b), bhi = __ldg(block_off + b + 1);
  const int64_t start = blo + G.w0;
  const int64_t n = min(bhi - start, (int64_t)1 << G.log_w);
  lo = start;
  len = n > 0 ? (int)n : 0;
}

// Units of work of a group: its chunks, cut into pieces of 2^log_u samples (at least 128) when there
// are fewer chunks than the CTA has warps, so that a group of few detectors and a long window still
// uses every warp.
__device__ __forceinline__ int unit_log(const PGroup& G, int warps) {
  int lu = G.log_w;
  while (lu > 7 && (G.n_blk << (G.log_w - lu)) < warps) lu--;
  return lu;
}
__device__ __forceinline__ void group_unit(const PGroup& G, const int64_t* __restrict__ block_off, int unit, int lu,
                                           int64_t& lo, int& len) {
  const int ls = G.log_w - lu;
  group_chunk(G, block_off, unit >> ls, lo, len);
  const int o = (unit & ((1 << ls) - 1)) << lu;
  lo += o;
  len = max(0, min(len - o, 1 << lu));
}

// Insert p into the set (bounded probing); returns the position, or -1 when the set is full.
__device__ __forceinline__ int set_insert(int32_t* keys, int32_t p, int* count) {
  uint32_t h = hash_of(p);
  for (int probe = 0; probe < kHash; probe++) {
    const int32_t prev = atomicCAS(keys + h, -1, p);
    if (prev == -1) {
      atomicAdd(count, 1);
      return (int)h;
    }
    if (prev == p) return (int)h;
    h = (h + 1) & (kHash - 1);
  }
  return -1;
}

__device__ __forceinline__ int set_find(const int32_t* keys, int32_t p) {
  uint32_t h = hash_of(p);
  for (int probe = 0; probe < kHash; probe++) {
    const int32_t k = keys[h];
    if (k == p) return (int)h;
    if (k == -1) return -1;
    h = (h + 1) & (kHash - 1);
  }
  return -1;
}

// Slot of the k-th smallest of a group's n pixels.  The lanes of a warp hold samples some pixels
// apart, along a sky row or across rows, so the ranks that one warp-wide access touches are often a
// multiple of 8 apart (a square focal plane scanned across its rows: 128); the low three bits of the
// rank are mixed with the higher ones so that such strides spread over the eight 16-byte bank groups
// (map windows read 19.6 shared wavefronts per 32 samples without it, 16 x 16 detectors, half of the
// intervals scanning along y).  A bijection on [0, n): the last partial group of 8 stays.
__device__ __forceinline__ int slot_of_rank(int k, int n) {
  return k < (n & ~7) ? (k & ~7) | ((k ^ (k >> 3) ^ (k >> 6) ^ (k >> 9)) & 7) : k;
}

// (cos x, sin x) for x in [-pi, pi] (the plan's reduced 2 psi)
__device__ __forceinline__ void weights_of_angle(float x, float& c, float& s) { __sincosf(x, &s, &c); }

}  // namespace

// Streaming arrays (slot, angle, TOD) are read and written with the evict-first cache policy
// (__ldcs / __stcs) so that they do not push the map, which the window gathers and the per-pixel
// atomics reuse, out of L2.

// One CTA per group.  Count mode (slot == nullptr): n_slots_out[g] = distinct kept pixels of the
// group, or -1 above kWinCap.  Fill mode: the pixel-sorted slot table and every sample's slot.
__global__ void __launch_bounds__(kWinThreads) k_win_build(const PGroup* __restrict__ groups,
                                                           const int64_t* __restrict__ block_off,
                                                           const int32_t* __restrict__ lpix,
                                                           int32_t* __restrict__ n_slots_out,
                                                           uint16_t* __restrict__ slot,
                                                           int32_t* __restrict__ slot_pix) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  int32_t* keys = reinterpret_cast<int32_t*>(smem_raw);                 // [kHash]
  int32_t* sorted = keys + kHash;                                       // [kWinCap]
  uint16_t* rank_of = reinterpret_cast<uint16_t*>(sorted + kWinCap);    // [kHash]
  __shared__ int s_count, s_n;
  const PGroup G = groups[blockIdx.x];
  for (int i = threadIdx.x; i < kHash; i += kWinThreads) keys[i] = -1;
  if (threadIdx.x == 0) {
    s_count = 0;
    s_n = 0;
  }
  __syncthreads();
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int lu = unit_log(G, kWarps), n_units = G.n_blk << (G.log_w - lu);
  for (int c = warp; c < n_units; c += kWarps) {
    int64_t lo;
    int len;
    group_unit(G, block_off, c, lu, lo, len);
    for (int o = lane; o < len; o += 32) {
      const int32_t p = __ldg(lpix + lo + o);
      if (p < 0) continue;
      if (*(volatile int*)&s_count > kWinCap) break;
      set_insert(keys, p, &s_count);
    }
  }
  __syncthreads();
  const int n = s_count;
  if (slot == nullptr) {
    if (threadIdx.x == 0) n_slots_out[blockIdx.x] = (n > kWinCap) ? -1 : n;
    return;
  }
  if (n != G.n_slots) {   // the host counted with the same kernel; a mismatch is a bug
    if (threadIdx.x == 0) atomicOr(n_slots_out, 1);
    return;
  }
  // compact the set and sort it (bitonic, padded to a power of two with INT_MAX)
  int n2 = 1;
  while (n2 < n) n2 <<= 1;
  for (int i = threadIdx.x; i < kHash; i += kWinThreads)
    if (keys[i] != -1) sorted[atomicAdd(&s_n, 1)] = keys[i];
  __syncthreads();
  for (int i = n + threadIdx.x; i < n2; i += kWinThreads) sorted[i] = 0x7fffffff;
  __syncthreads();
  for (int k = 2; k <= n2; k <<= 1) {
    for (int j = k >> 1; j > 0; j >>= 1) {
      for (int i = threadIdx.x; i < n2; i += kWinThreads) {
        const int l = i ^ j;
        if (l > i) {
          const int32_t a = sorted[i], b = sorted[l];
          const bool up = (i & k) == 0;
          if ((a > b) == up) {
            sorted[i] = b;
            sorted[l] = a;
          }
        }
      }
      __syncthreads();
    }
  }
  for (int k = threadIdx.x; k < n; k += kWinThreads) {
    const int32_t p = sorted[k];
    const int sl = slot_of_rank(k, n);
    slot_pix[G.slot_off + sl] = p;
    const int h = set_find(keys, p);
    if (h >= 0) rank_of[h] = (uint16_t)sl;
  }
  __syncthreads();
  for (int c = warp; c < n_units; c += kWarps) {
    int64_t lo;
    int len;
    group_unit(G, block_off, c, lu, lo, len);
    for (int o = lane; o < len; o += 32) {
      const int32_t p = __ldg(lpix + lo + o);
      uint16_t r = kNoSlot;
      if (p >= 0) {
        const int h = set_find(keys, p);
        if (h >= 0) r = rank_of[h];
      }
      slot[lo + o] = r;
    }
  }
}

constexpr size_t kBuildSmem = (size_t)kHash * 4 + (size_t)kWinCap * 4 + (size_t)kHash * 2;

#define MM_TRY_CUDA(expr)             \
  do {                                \
    const cudaError_t e_ = (expr);    \
    if (e_ != cudaSuccess) return e_; \
  } while (0)

// dynamic shared-memory limit of a kernel, set once per process
template <typename K>
static cudaError_t smem_limit_once(K kernel, size_t bytes, cudaError_t& status, bool& done) {
  if (!done) {
    status = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
    done = true;
  }
  return status;
}

cudaError_t launch_win_build(const PGroup* groups, int64_t n_groups, const int64_t* block_off,
                             const int32_t* lpix, int32_t* n_slots_out, uint16_t* slot, int32_t* slot_pix,
                             cudaStream_t s) {
  if (n_groups == 0) return cudaSuccess;
  if (n_groups > 0x7fffffffLL) return cudaErrorInvalidConfiguration;
  static cudaError_t st = cudaSuccess;
  static bool set = false;
  MM_TRY_CUDA(smem_limit_once(k_win_build, kBuildSmem, st, set));
  k_win_build<<<(unsigned)n_groups, kWinThreads, kBuildSmem, s>>>(groups, block_off, lpix, n_slots_out, slot,
                                                                   slot_pix);
  return cudaGetLastError();
}

// ---- sorted entries of the groups (P^T by run sums) -------------------------------------------
// One CTA per group: a counting sort of its kept samples by slot in shared memory, written out in
// the interleaved blocks that k_point_sorted reads.
__global__ void __launch_bounds__(kWinThreads) k_srt_build(const PGroup* __restrict__ groups,
                                                           const int64_t* __restrict__ block_off,
                                                           const uint16_t* __restrict__ slot,
                                                           const float* __restrict__ ang2, uint16_t* __restrict__ ent,
                                                           float* __restrict__ ent_ang,
                                                           uint16_t* __restrict__ first_slot) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  int32_t* off = reinterpret_cast<int32_t*>(smem_raw);                  // [kWinCap + 1] counts, then next positions
  uint32_t* key = reinterpret_cast<uint32_t*>(off + kWinCap + 4);       // [kWinMaxSamples] slot << 16 | position
  __shared__ int32_t warp_sum[kWarps];
  const PGroup G = groups[blockIdx.x];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int row = srt_row(G.log_w), zero = G.n_blk * row;
  const int lu = unit_log(G, kWarps), n_units = G.n_blk << (G.log_w - lu), ls = G.log_w - lu;
  for (int i = tid; i <= kWinCap; i += kWinThreads) off[i] = 0;
  __syncthreads();
  for (int u = warp; u < n_units; u += kWarps) {
    int64_t lo;
    int len;
    group_unit(G, block_off, u, lu, lo, len);
    for (int o = lane; o < len; o += 32) {
      const uint32_t s = slot[lo + o];
      if (s != kNoSlot) atomicAdd(off + s, 1);
    }
  }
  __syncthreads();
  // exclusive scan of the counts: kWinCap / kWinThreads consecutive slots per thread
  constexpr int kPer = kWinCap / kWinThreads;
  int32_t c[kPer], sum = 0;
#pragma unroll
  for (int i = 0; i < kPer; i++) {
    c[i] = off[tid * kPer + i];
    sum += c[i];
  }
  int32_t inc = sum;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int32_t t = __shfl_up_sync(0xffffffffu, inc, o);
    if (lane >= o) inc += t;
  }
  if (lane == 31) warp_sum[warp] = inc;
  __syncthreads();
  int32_t base = inc - sum, total = 0;
  for (int w = 0; w < kWarps; w++) {
    if (w < warp) base += warp_sum[w];
    total += warp_sum[w];
  }
#pragma unroll
  for (int i = 0; i < kPer; i++) {
    off[tid * kPer + i] = base;
    base += c[i];
  }
  __syncthreads();
  for (int u = warp; u < n_units; u += kWarps) {
    int64_t lo, lo0;
    int len, len0;
    group_unit(G, block_off, u, lu, lo, len);
    group_chunk(G, block_off, u >> ls, lo0, len0);
    const int pos0 = (u >> ls) * row + (int)(lo0 & 3) + (int)(lo - lo0);
    for (int o = lane; o < len; o += 32) {
      const uint32_t s = slot[lo + o];
      if (s != kNoSlot) key[atomicAdd(off + s, 1)] = (s << 16) | (uint32_t)(pos0 + o);
    }
  }
  __syncthreads();
  for (int i = tid; i < G.n_srt * kSrtBlock; i += kWinThreads) {
    const int b = i / kSrtBlock, l = (i / 32) % 32, e = i % 32;
    uint32_t w = (uint32_t)zero;
    float a = 0.f;
    if (i < total) {
      const uint32_t k = key[i], pos = k & 0xFFFFu;
      w = pos | ((e > 0 && (key[i - 1] >> 16) != (k >> 16)) ? kSrtRun : 0u);
      const int r = (int)pos / row;
      int64_t lo;
      int len;
      group_chunk(G, block_off, r, lo, len);
      a = __ldg(ang2 + lo + ((int)pos - r * row - (int)(lo & 3)));
    }
    const int64_t blk = (G.srt_off + b) * kSrtBlock;
    ent[blk + (e / 8) * 256 + l * 8 + e % 8] = (uint16_t)w;
    ent_ang[blk + (e / 4) * 128 + l * 4 + e % 4] = a;
    if (e == 0) first_slot[(G.srt_off + b) * 32 + l] = i < total ? (uint16_t)(key[i] >> 16) : kNoSlot;
  }
}

constexpr size_t kSrtBuildSmem = (size_t)(kWinCap + 4) * 4 + (size_t)kWinMaxSamples * 4;
cudaError_t launch_srt_build(const PGroup* groups, int64_t n_groups, const int64_t* block_off, const uint16_t* slot,
                             const float* ang2, uint16_t* ent, float* ent_ang, uint16_t* first_slot, cudaStream_t s) {
  if (n_groups == 0) return cudaSuccess;
  if (n_groups > 0x7fffffffLL) return cudaErrorInvalidConfiguration;
  static cudaError_t st = cudaSuccess;
  static bool set = false;
  MM_TRY_CUDA(smem_limit_once(k_srt_build, kSrtBuildSmem, st, set));
  k_srt_build<<<(unsigned)n_groups, kWinThreads, kSrtBuildSmem, s>>>(groups, block_off, slot, ang2, ent, ent_ang,
                                                                    first_slot);
  return cudaGetLastError();
}

// ---- chunk walking shared by the un-point and point kernels ------------------------------------
// A warp takes CPI = 32 / LPC chunks at a time, LPC = min(32, W / 4) lanes per chunk.  Inside a
// chunk [lo, lo + len) the lanes walk aligned quads of 4 samples [a0, a1) (a0 = lo rounded up to
// 4) with vector loads; the at most 3 + 3 samples before a0 and after a1 go one per lane.
struct ChunkWalk {
  int lpc, cpi, sub, ql;
};
__device__ __forceinline__ ChunkWalk chunk_walk(int log_u, int lane) {
  ChunkWalk w;
  w.lpc = log_u >= 7 ? 32 : (1 << (log_u - 2));
  w.cpi = 32 / w.lpc;
  w.sub = lane / w.lpc;
  w.ql = lane % w.lpc;
  return w;
}

// Visit every sample of unit c (pieces of 2^lu samples): f_quad(base, q4) for aligned quads (samples
// base + 4 q4 .. + 3), f_one(i) for the single samples of the ragged ends.  Global sample indices are 64-bit.
template <typename FQ, typename F1>
__device__ __forceinline__ void visit_unit(const PGroup& G, const int64_t* __restrict__ block_off, int c, int lu,
                                           const ChunkWalk& w, FQ f_quad, F1 f_one) {
  int64_t lo;
  int len;
  group_unit(G, block_off, c, lu, lo, len);
  if (len <= 0) return;
  const int64_t a0 = (lo + 3) & ~(int64_t)3;
  const int head = (int)min((int64_t)len, a0 - lo);
  const int nq = (len - head) >> 2;
  const int tail = len - head - 4 * nq;
  const int64_t a1 = a0 + 4 * (int64_t)nq;
  if (w.ql < head) f_one(lo + w.ql);
  if (w.ql < tail) f_one(a1 + w.ql);
  for (int q = w.ql; q < nq; q += w.lpc) f_quad(a0, q);
}

// Pointing loads (slot, angle): evict-first when a pass has one column; with several columns the
// CTA reads the same group's pointing once per column, so it is kept in L2 for the later ones.
template <typename T>
__device__ __forceinline__ T ld_point(const T* p, bool keep) { return keep ? __ldg(p) : __ldcs(p); }

// Padded shared-memory index of slot k's accumulators.  A lane holds 4 consecutive samples, so one warp-wide
// access touches slots about 4 x (pixels per sample) apart; one padding word per 32 scalar slots
// keeps strides of 1, 2, 4 and 8 slots in distinct banks.
__device__ __forceinline__ int acc_index(int k) { return k + (k >> 5); }
constexpr int kAccStride = kWinCap + kWinCap / 32;

// Rows of a group (one per detector chunk) in shared memory: first sample and length, 12 bytes a row.
struct RowTab {
  int64_t* lo;
  int32_t* len;
  __device__ RowTab(void* base, int dets) : lo(reinterpret_cast<int64_t*>(base)), len(reinterpret_cast<int32_t*>(lo + dets)) {}
  __device__ __forceinline__ void load(const PGroup& G, const int64_t* __restrict__ block_off) {
    for (int c = threadIdx.x; c < G.n_blk; c += blockDim.x) {
      int64_t l;
      int n;
      group_chunk(G, block_off, c, l, n);
      lo[c] = l;
      len[c] = n;
    }
  }
};
static size_t row_tab_bytes(int dets) { return (size_t)dets * 12; }

// Aligned quads of a group's rows: a warp takes 128 samples at a time, LPC = min(32, W / 4) lanes per
// row, quad q of a row being samples [lo - lo % 4 + 4 q, + 4).  A row that does not start on a multiple
// of 4 has one quad more, W / 4, which is visited apart.
struct QuadWalk {
  int lu, ls, lpc, cpi, sub, ql, n_units;
};
__device__ __forceinline__ QuadWalk quad_walk(const PGroup& G, int lane) {
  QuadWalk w;
  w.lu = min(G.log_w, 7);
  w.ls = G.log_w - w.lu;
  w.lpc = 1 << (w.lu - 2);
  w.cpi = 32 / w.lpc;
  w.sub = lane / w.lpc;
  w.ql = lane % w.lpc;
  w.n_units = G.n_blk << w.ls;
  return w;
}

// The group's map entries into shared memory by asynchronous 16-byte copies: all gathers of a thread are
// in flight at once (with loads through registers the fill took 34 of 175 us, 67M samples).
__device__ __forceinline__ void fill_window(float4* win, const float4* __restrict__ x, const int32_t* __restrict__ pix,
                                            int n_slots) {
  constexpr int U = 8;
  for (int k0 = threadIdx.x; k0 < n_slots; k0 += U * blockDim.x) {
    int32_t p[U];
#pragma unroll
    for (int j = 0; j < U; j++) {
      const int k = k0 + j * blockDim.x;
      p[j] = k < n_slots ? __ldg(pix + k) : -1;
    }
#pragma unroll
    for (int j = 0; j < U; j++)
      if (p[j] >= 0)
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(
                         (uint32_t)__cvta_generic_to_shared(win + k0 + j * blockDim.x)),
                     "l"(x + p[j])
                     : "memory");
  }
}

// t = P x over the windows: one CTA per group, the group's map entries of column r in shared
// memory, then one coalesced pass over the group's samples, each lane's next slots and angles loaded
// while it works on the current ones (and the first before the window is filled).  Bound by HBM:
// 10 B per sample (slot 2, angle 4, t 4); 256 detectors x 4 x 65,536 samples: 144 us, 4.7 TB/s (175 us
// before the window was filled by asynchronous copies, 4 x 65,536 samples: 55 -> 5 us).  Several columns are
// bound by instruction issue (slots, angles and cos / sin again for each), so NC = 2 of them go through the
// samples together while two windows leave four CTAs on an SM: 8.4M samples x 16 columns, 205 -> 156 us.
// MULTI: the group's problem (one column) comes from probs[G.prob].
constexpr int kUnpointThreads = 256;
template <bool MULTI, int NC>
__global__ void __launch_bounds__(kUnpointThreads, NC == 1 ? 6 : 4) k_unpoint_win32(
    const PGroup* __restrict__ groups, const int64_t* __restrict__ block_off,
    const uint16_t* __restrict__ slot, const int32_t* __restrict__ slot_pix, const float* __restrict__ ang2,
    const float4* __restrict__ x4, int64_t x_stride4, int nrhs, const int32_t* __restrict__ done,
    int done_stride, float* __restrict__ t, int64_t t_stride, const WinProb* __restrict__ probs, WinSize size) {
  extern __shared__ float4 win[];   // [NC][size.slots], then the row table
  RowTab rt(win + NC * size.slots, size.dets);
  const PGroup G = groups[blockIdx.x];
  if constexpr (MULTI) {
    const WinProb& pp = probs[G.prob];
    block_off = pp.block_off;
    slot = pp.slot;
    slot_pix = pp.slot_pix;
    ang2 = pp.ang2;
    x4 = reinterpret_cast<const float4*>(pp.x);
    t = pp.t;
    done = pp.done;
  }
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, warps = blockDim.x >> 5;
  const QuadWalk w = quad_walk(G, lane);
  const bool keep = nrhs > NC;
  rt.load(G, block_off);
  __syncthreads();
  for (int r = 0; r < nrhs; r += NC) {
    bool on[NC], any = false;
#pragma unroll
    for (int c = 0; c < NC; c++) {
      on[c] = r + c < nrhs && (done == nullptr || done[(int64_t)(r + c) * done_stride] == 0);
      any |= on[c];
    }
    if (!any) continue;
    // the columns' values of a sample
    auto value = [&](uint32_t sl, float a, float (&v)[NC]) {
#pragma unroll
      for (int c = 0; c < NC; c++) v[c] = 0.f;
      if (sl == kNoSlot) return;
      float cs, sn;
      weights_of_angle(a, cs, sn);
#pragma unroll
      for (int c = 0; c < NC; c++) {
        const float4 m = win[c * size.slots + sl];
        v[c] = m.x + cs * m.y + sn * m.z;
      }
    };
    // quad q of row c: its samples and the ones of them inside the row, [e0, e1); a sample outside it is a
    // neighbouring row's (of any group: its slot is below size.slots too) or past the end (kNoSlot)
    struct Quad {
      int64_t i;
      int e0, e1;
      uint2 s;
      float4 a;
    };
    auto load = [&](int c, int q, Quad& d) {
      const int64_t lo = rt.lo[c];
      const int a = (int)(lo & 3), end = a + rt.len[c];
      d.i = lo - a + 4 * (int64_t)q;
      d.e0 = q == 0 ? a : 0;
      d.e1 = min(4, end - 4 * q);
      if (d.e1 > d.e0) {
        d.s = ld_point(reinterpret_cast<const uint2*>(slot + d.i), keep);
        d.a = ld_point(reinterpret_cast<const float4*>(ang2 + d.i), keep);
      }
    };
    auto emit = [&](const Quad& d) {
      if (d.e1 <= d.e0) return;
      float v0[NC], v1[NC], v2[NC], v3[NC];
      value(d.s.x & 0xFFFFu, d.a.x, v0);
      value(d.s.x >> 16, d.a.y, v1);
      value(d.s.y & 0xFFFFu, d.a.z, v2);
      value(d.s.y >> 16, d.a.w, v3);
#pragma unroll
      for (int c = 0; c < NC; c++) {
        if (!on[c]) continue;
        float* to = t + (r + c) * t_stride + d.i;
        if (d.e1 - d.e0 == 4) {
          __stcs(reinterpret_cast<float4*>(to), make_float4(v0[c], v1[c], v2[c], v3[c]));
        } else {
          if (d.e0 <= 0 && d.e1 > 0) __stcs(to, v0[c]);
          if (d.e0 <= 1 && d.e1 > 1) __stcs(to + 1, v1[c]);
          if (d.e0 <= 2 && d.e1 > 2) __stcs(to + 2, v2[c]);
          if (d.e0 <= 3 && d.e1 > 3) __stcs(to + 3, v3[c]);
        }
      }
    };
    auto load_unit = [&](int u, Quad& d) {
      d.e0 = d.e1 = 0;
      if (u < w.n_units) load(u >> w.ls, ((u & ((1 << w.ls) - 1)) << (w.lu - 2)) + w.ql, d);
    };
    Quad cur, nxt;
    const int step = warps * w.cpi;
    int u = warp * w.cpi + w.sub;
    load_unit(u, cur);
    if (r > 0) __syncthreads();   // the previous column's window is no longer read
#pragma unroll
    for (int c = 0; c < NC; c++)
      if (on[c]) fill_window(win + c * size.slots, x4 + (r + c) * x_stride4, slot_pix + G.slot_off, G.n_slots);
    asm volatile("cp.async.wait_all;" ::: "memory");
    __syncthreads();
    for (; u < w.n_units; u += step) {
      load_unit(u + step, nxt);
      emit(cur);
      cur = nxt;
    }
    for (int c = threadIdx.x; c < G.n_blk; c += blockDim.x) {   // the last quad of rows off a multiple of 4
      if ((int)(rt.lo[c] & 3) + rt.len[c] > (1 << G.log_w)) {
        load(c, 1 << (G.log_w - 2), cur);
        emit(cur);
      }
    }
  }
}
constexpr size_t kUnpointSmem = (size_t)kWinCap * sizeof(float4) + 512 * 12;   // most of any group

static int unpoint_threads(const WinSize& z) { return std::min(z.threads, kUnpointThreads); }
static size_t unpoint_smem(const WinSize& z, int nc) { return (size_t)nc * z.slots * sizeof(float4) + row_tab_bytes(z.dets); }
constexpr size_t kUnpointPairSmem = 56 * 1024;   // four CTAs of column pairs on an SM

cudaError_t launch_unpoint_win32(const PGroup* groups, int64_t n_groups, const WinSize& size, const int64_t* block_off,
                                 const uint16_t* slot, const int32_t* slot_pix, const float* ang2,
                                 const float* x4, int64_t x_stride, int nrhs, const int32_t* done,
                                 int done_stride, float* t, int64_t t_stride, cudaStream_t s) {
  if (n_groups == 0 || nrhs <= 0) return cudaSuccess;
  if (n_groups > 0x7fffffffLL || t_stride % 4 != 0) return cudaErrorInvalidValue;
  static cudaError_t st = cudaSuccess;
  static bool set = false;
  if (nrhs > 1 && unpoint_smem(size, 2) <= kUnpointPairSmem) {
    static cudaError_t st2 = cudaSuccess;
    static bool set2 = false;
    MM_TRY_CUDA(smem_limit_once(k_unpoint_win32<false, 2>, kUnpointPairSmem, st2, set2));
    k_unpoint_win32<false, 2><<<(unsigned)n_groups, unpoint_threads(size), unpoint_smem(size, 2), s>>>(
        groups, block_off, slot, slot_pix, ang2, reinterpret_cast<const float4*>(x4), x_stride / 4, nrhs, done,
        done_stride, t, t_stride, nullptr, size);
    return cudaGetLastError();
  }
  MM_TRY_CUDA(smem_limit_once(k_unpoint_win32<false, 1>, kUnpointSmem, st, set));
  k_unpoint_win32<false, 1><<<(unsigned)n_groups, unpoint_threads(size), unpoint_smem(size, 1), s>>>(
      groups, block_off, slot, slot_pix, ang2, reinterpret_cast<const float4*>(x4), x_stride / 4, nrhs, done,
      done_stride, t, t_stride, nullptr, size);
  return cudaGetLastError();
}

cudaError_t launch_unpoint_win32_multi(const PGroup* groups, int64_t n_groups, const WinSize& size, const WinProb* probs,
                                       cudaStream_t s) {
  if (n_groups == 0) return cudaSuccess;
  if (n_groups > 0x7fffffffLL || probs == nullptr) return cudaErrorInvalidValue;
  static cudaError_t st = cudaSuccess;
  static bool set = false;
  MM_TRY_CUDA(smem_limit_once(k_unpoint_win32<true, 1>, kUnpointSmem, st, set));
  k_unpoint_win32<true, 1><<<(unsigned)n_groups, unpoint_threads(size), unpoint_smem(size, 1), s>>>(
      groups, nullptr, nullptr, nullptr, nullptr, nullptr, 0, 1, nullptr, 0, nullptr, 0, probs, size);
  return cudaGetLastError();
}

// The map that this CTA's group adds to (PtMaps), y4 or one of the extra ones of `stride4` pixels.
__device__ __forceinline__ float4* group_map(float4* y4, int64_t stride4, const PtMaps& maps) {
  const int k = blockIdx.x & (maps.n - 1);
  return k == 0 ? y4 : reinterpret_cast<float4*>(maps.extra) + (k - 1) * stride4;
}

__global__ void k_sum_maps(PtMaps maps, int64_t stride4, const int32_t* __restrict__ done, int done_stride,
                           float4* __restrict__ y4, int64_t n) {
  if (done != nullptr && done[(int64_t)blockIdx.y * done_stride] != 0) return;
  const int64_t col = blockIdx.y * n;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    float4 v = y4[col + i];
    for (int k = 1; k < maps.n; k++) {
      const float4 e = __ldcs(reinterpret_cast<const float4*>(maps.extra) + (k - 1) * stride4 + col + i);
      v.x += e.x;
      v.y += e.y;
      v.z += e.z;
    }
    y4[col + i] = v;
  }
}
cudaError_t launch_sum_maps(const PtMaps& maps, int nrhs, const int32_t* done, int done_stride, float* y4,
                            int64_t y_stride, cudaStream_t s) {
  const int64_t n = y_stride / 4;
  if (maps.n <= 1 || n == 0 || nrhs <= 0) return cudaSuccess;
  const dim3 grid((unsigned)std::min<int64_t>((n + 255) / 256, 8 * (int64_t)sm_count()), nrhs);
  k_sum_maps<<<grid, 256, 0, s>>>(maps, nrhs * n, done, done_stride, reinterpret_cast<float4*>(y4), n);
  return cudaGetLastError();
}

// y += P^T u by run sums: one CTA per group.  The group's u goes to shared memory by 16-byte
// asynchronous copies; then every lane walks 32 consecutive pixel-sorted entries (position, angle),
// sums u, u cos 2psi, u sin 2psi of a run of equal pixels in registers and adds each run to the map
// with one float4 atomic (a pixel's sum arrives in one piece except where a lane's range cuts it).
// Bound by HBM: 10 B per sample (entry 2, angle 4, u 4).  The three FP32 shared-memory additions per
// sample that it replaces are loops of compare-and-swap on this machine and kept the shared-memory pipe
// at 83 to 87% (20 shared wavefronts per 32 samples, here 4): 256 detectors x 4 x 524,288 samples 1.52
// -> 1.08 ms, 64 x 262,144 64 -> 42 us, 4 x 65,536 86 -> 8 us (with the groups of build_windows).
// Several columns: NC = 2 of them share the entries, angles, cos / sin and pixels of the runs while both
// columns' u leave two CTAs on an SM (8.4M samples x 16 columns: 223 -> 201 us).
template <bool MULTI, int NC>
__global__ void __launch_bounds__(kWinThreads, 2) k_point_sorted(
    const PGroup* __restrict__ groups, const int64_t* __restrict__ block_off, const uint4* __restrict__ ent,
    const float4* __restrict__ ent_ang, const uint16_t* __restrict__ first_slot,
    const int32_t* __restrict__ slot_pix, const float* __restrict__ u, int64_t u_stride, int nrhs,
    const int32_t* __restrict__ done, int done_stride, float4* __restrict__ y4, int64_t y_stride4,
    const WinProb* __restrict__ probs, WinSize size, PtMaps maps) {
  extern __shared__ __align__(16) float us[];   // [NC][size.rows]: n_blk rows of W + 4, then a zero; the row table
  const PGroup G = groups[blockIdx.x];
  if constexpr (MULTI) {
    const WinProb& pp = probs[G.prob];
    block_off = pp.block_off;
    ent = pp.srt_ent;
    ent_ang = pp.srt_ang;
    first_slot = pp.srt_slot;
    slot_pix = pp.slot_pix;
    u = pp.u;
    y4 = group_map(reinterpret_cast<float4*>(pp.y), pp.n_obs, pp.maps);
    done = pp.done;
  } else {
    y4 = group_map(y4, nrhs * y_stride4, maps);
  }
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, warps = blockDim.x >> 5;
  const int row = srt_row(G.log_w);
  const QuadWalk w = quad_walk(G, lane);
  RowTab rt(us + NC * size.rows, size.dets);
  const int32_t* __restrict__ pix = slot_pix + G.slot_off;
  rt.load(G, block_off);
  for (int r = 0; r < nrhs; r += NC) {
    bool on[NC], any = false;
#pragma unroll
    for (int c = 0; c < NC; c++) {
      on[c] = r + c < nrhs && (done == nullptr || done[(int64_t)(r + c) * done_stride] == 0);
      any |= on[c];
    }
    if (!any) continue;
    // this warp's first block of entries and half of its angles, on their way during the staging
    uint4 e[4];
    float4 a[4];
    int sl = kNoSlot;
    if (warp < G.n_srt) {
      const int64_t blk = G.srt_off + warp;
      sl = __ldg(first_slot + blk * 32 + lane);
#pragma unroll
      for (int o = 0; o < 4; o++) {
        e[o] = __ldg(ent + blk * (kSrtBlock / 8) + o * 32 + lane);
        a[o] = __ldg(ent_ang + blk * (kSrtBlock / 4) + o * 32 + lane);
      }
    }
    __syncthreads();   // the rows are there, the previous column's u is no longer read
    auto copy = [&](int c, int q) {
      const int64_t lo = rt.lo[c];
      const int a0 = (int)(lo & 3), len = rt.len[c];
      if (len > 0 && 4 * q < a0 + len) {
#pragma unroll
        for (int k = 0; k < NC; k++)
          if (on[k])
            asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(
                             (uint32_t)__cvta_generic_to_shared(us + k * size.rows + c * row + 4 * q)),
                         "l"(u + (r + k) * u_stride + lo - a0 + 4 * q)
                         : "memory");
      }
    };
    for (int c0 = warp * w.cpi + w.sub; c0 < w.n_units; c0 += warps * w.cpi)
      copy(c0 >> w.ls, ((c0 & ((1 << w.ls) - 1)) << (w.lu - 2)) + w.ql);
    for (int c = threadIdx.x; c < G.n_blk; c += blockDim.x) copy(c, 1 << (G.log_w - 2));
    if (threadIdx.x < NC) us[threadIdx.x * size.rows + G.n_blk * row] = 0.f;
    asm volatile("cp.async.commit_group;\ncp.async.wait_all;" ::: "memory");
    __syncthreads();
    float4* yr = y4 + r * y_stride4;
    for (int b = warp; b < G.n_srt; b += warps) {
      const int64_t blk = G.srt_off + b;
      const uint4* ep = ent + blk * (kSrtBlock / 8) + lane;
      const float4* ap = ent_ang + blk * (kSrtBlock / 4) + lane;
      if (b != warp) {
        sl = __ldg(first_slot + blk * 32 + lane);
#pragma unroll
        for (int o = 0; o < 4; o++) {
          e[o] = __ldg(ep + o * 32);
          a[o] = __ldg(ap + o * 32);
        }
      }
      if (sl == kNoSlot) continue;
      int32_t p = __ldg(pix + sl);
      float s0[NC], s1[NC], s2[NC];
#pragma unroll
      for (int k = 0; k < NC; k++) s0[k] = s1[k] = s2[k] = 0.f;
      auto add_run = [&]() {
#pragma unroll
        for (int k = 0; k < NC; k++)
          if (on[k]) atomicAdd(yr + k * y_stride4 + p, make_float4(s0[k], s1[k], s2[k], 0.f));
      };
      auto one = [&](uint32_t en, float an) {
        if (en & kSrtRun) {   // a new run: the previous pixel's sum is complete
          add_run();
          p = __ldg(pix + ++sl);
#pragma unroll
          for (int k = 0; k < NC; k++) s0[k] = s1[k] = s2[k] = 0.f;
        }
        float cs, sn;
        weights_of_angle(an, cs, sn);
#pragma unroll
        for (int k = 0; k < NC; k++) {
          const float y = us[k * size.rows + (en & 0x7FFFu)];
          s0[k] += y;
          s1[k] = fmaf(cs, y, s1[k]);
          s2[k] = fmaf(sn, y, s2[k]);
        }
      };
#pragma unroll
      for (int o = 0; o < 4; o++) {
        // angle quads 2 o and 2 o + 1: four are held, the next two are loaded as these are used
        const int h = (2 * o) & 3;
        const float4 a0 = a[h], a1 = a[h + 1];
        if (o < 2) {
          a[h] = __ldg(ap + (2 * o + 4) * 32);
          a[h + 1] = __ldg(ap + (2 * o + 5) * 32);
        }
        one(e[o].x & 0xFFFFu, a0.x);
        one(e[o].x >> 16, a0.y);
        one(e[o].y & 0xFFFFu, a0.z);
        one(e[o].y >> 16, a0.w);
        one(e[o].z & 0xFFFFu, a1.x);
        one(e[o].z >> 16, a1.y);
        one(e[o].w & 0xFFFFu, a1.z);
        one(e[o].w >> 16, a1.w);
      }
      add_run();
    }
  }
}

constexpr int kPointPairSmem = 112 * 1024;   // two CTAs of column pairs on an SM
static cudaError_t point_sorted_attr() {
  constexpr int kMost = (kWinMaxSamples / 32 * ((1 << 5) + 4) + 4) * (int)sizeof(float) + 512 * 12;
  static const cudaError_t e = [] {
    cudaError_t r = cudaFuncSetAttribute(k_point_sorted<false, 1>, cudaFuncAttributeMaxDynamicSharedMemorySize, kMost);
    if (r == cudaSuccess)
      r = cudaFuncSetAttribute(k_point_sorted<false, 2>, cudaFuncAttributeMaxDynamicSharedMemorySize, kPointPairSmem);
    if (r == cudaSuccess)
      r = cudaFuncSetAttribute(k_point_sorted<true, 1>, cudaFuncAttributeMaxDynamicSharedMemorySize, kMost);
    return r;
  }();
  return e;
}
static size_t point_sorted_smem(const WinSize& z, int nc) { return (size_t)nc * z.rows * sizeof(float) + row_tab_bytes(z.dets); }
static int point_sorted_threads(const WinSize& z) { return 32 * std::min(kWinThreads / 32, std::max(1, z.blocks)); }

cudaError_t launch_point_sorted(const PGroup* groups, int64_t n_groups, const WinSize& size,
                                const int64_t* block_off, const uint16_t* ent, const float* ent_ang,
                                const uint16_t* first_slot, const int32_t* slot_pix, const float* u,
                                int64_t u_stride, int nrhs, const int32_t* done, int done_stride, float* y4,
                                int64_t y_stride, const PtMaps& maps, cudaStream_t s) {
  if (n_groups == 0 || nrhs <= 0) return cudaSuccess;
  if (n_groups > 0x7fffffffLL || u_stride % 4 != 0) return cudaErrorInvalidValue;
  MM_TRY_CUDA(point_sorted_attr());
  const bool pair = nrhs > 1 && point_sorted_smem(size, 2) <= (size_t)kPointPairSmem;
  auto* kernel = pair ? k_point_sorted<false, 2> : k_point_sorted<false, 1>;
  kernel<<<(unsigned)n_groups, point_sorted_threads(size), point_sorted_smem(size, pair ? 2 : 1), s>>>(
      groups, block_off, reinterpret_cast<const uint4*>(ent), reinterpret_cast<const float4*>(ent_ang), first_slot,
      slot_pix, u, u_stride, nrhs, done, done_stride, reinterpret_cast<float4*>(y4), y_stride / 4, nullptr, size,
      maps);
  return cudaGetLastError();
}

cudaError_t launch_point_sorted_multi(const PGroup* groups, int64_t n_groups, const WinSize& size,
                                      const WinProb* probs, cudaStream_t s) {
  if (n_groups == 0) return cudaSuccess;
  if (n_groups > 0x7fffffffLL || probs == nullptr) return cudaErrorInvalidValue;
  MM_TRY_CUDA(point_sorted_attr());
  k_point_sorted<true, 1><<<(unsigned)n_groups, point_sorted_threads(size), point_sorted_smem(size, 1), s>>>(
      groups, nullptr, nullptr, nullptr, nullptr, nullptr, nullptr, 0, 1, nullptr, 0, nullptr, 0, probs, size, PtMaps{});
  return cudaGetLastError();
}

// ---- P^T by segment reduction over pixel-sorted sub-windows ----------------------------------
// Sample l = c 2^log_s + o of sub-window sw: global index, false past its chunk's end.
__device__ __forceinline__ bool sub_sample(const PGroup& G, const int64_t* __restrict__ block_off, int sw,
                                           int log_s, int l, int64_t& i) {
  int64_t lo;
  int len;
  group_chunk(G, block_off, l >> log_s, lo, len);
  const int o = (sw << log_s) + (l & ((1 << log_s) - 1));
  i = lo + o;
  return o < len;
}

// One CTA per group: for each sub-window, the keys (slot << 16 | l) of its samples (masked ones
// with slot kNoSlot) sorted ascending in shared memory (bitonic, padded with 0xFFFFFFFF), so equal
// slots form runs ordered by l, then written out with each kept entry's angle.
__global__ void __launch_bounds__(kWinThreads) k_seg_build(const PGroup* __restrict__ groups,
                                                           const int64_t* __restrict__ block_off,
                                                           const uint16_t* __restrict__ slot,
                                                           const float* __restrict__ ang2, int sub_cap,
                                                           uint32_t* __restrict__ ent,
                                                           float* __restrict__ ent_ang,
                                                           int32_t* __restrict__ kept) {
  extern __shared__ __align__(16) uint32_t keys[];   // [next power of two >= sub_cap]
  __shared__ int s_kept;
  const PGroup G = groups[blockIdx.x];
  const int ls = seg_log_s(G.n_blk, G.log_w, sub_cap);
  const int n_sub = 1 << (G.log_w - ls);
  const int64_t stride = seg_stride(G.n_blk, ls);
  const int n_l = G.n_blk << ls;
  int n2 = 1;
  while (n2 < n_l) n2 <<= 1;
  for (int sw = 0; sw < n_sub; sw++) {
    if (threadIdx.x == 0) s_kept = 0;
    __syncthreads();
    int my_kept = 0;
    for (int l = threadIdx.x; l < n2; l += kWinThreads) {
      uint32_t key = 0xFFFFFFFFu;
      if (l < n_l) {
        int64_t i;
        uint32_t sl = kNoSlot;
        if (sub_sample(G, block_off, sw, ls, l, i)) sl = slot[i];
        key = (sl << 16) | (uint32_t)l;
        my_kept += sl != kNoSlot;
      }
      keys[l] = key;
    }
    atomicAdd(&s_kept, my_kept);
    __syncthreads();
    for (int k = 2; k <= n2; k <<= 1) {
      for (int j = k >> 1; j > 0; j >>= 1) {
        for (int i = threadIdx.x; i < n2; i += kWinThreads) {
          const int l = i ^ j;
          if (l > i) {
            const uint32_t a = keys[i], b = keys[l];
            if ((a > b) == ((i & k) == 0)) {
              keys[i] = b;
              keys[l] = a;
            }
          }
        }
        __syncthreads();
      }
    }
    const int nk = s_kept;
    const int64_t base = G.ent_off + (int64_t)sw * stride;
    for (int j = threadIdx.x; j < stride; j += kWinThreads) {
      uint32_t e = (uint32_t)kNoSlot << 16;
      float a = 0.f;
      if (j < nk) {
        e = keys[j];
        int64_t i;
        sub_sample(G, block_off, sw, ls, (int)(e & 0xFFFFu), i);
        a = __ldg(ang2 + i);
      }
      ent[base + j] = e;
      ent_ang[base + j] = a;
    }
    if (threadIdx.x == 0) kept[G.sub0 + sw] = nk;
    __syncthreads();   // the keys are rewritten by the next sub-window
  }
}

constexpr int kSegSubMax = 16384;
constexpr size_t kSegBuildSmemMax = (size_t)kSegSubMax * sizeof(uint32_t);
constexpr size_t kPointSegSmemMax = (size_t)3 * kAccStride * sizeof(float) + (size_t)kSegSubMax * sizeof(float);

static int pow2_at_least(int n) {
  int p = 1;
  while (p < n) p <<= 1;
  return p;
}

cudaError_t launch_seg_build(const PGroup* groups, int64_t n_groups, const int64_t* block_off,
                             const uint16_t* slot, const float* ang2, int sub_cap, uint32_t* ent,
                             float* ent_ang, int32_t* kept, cudaStream_t s) {
  if (n_groups == 0) return cudaSuccess;
  if (n_groups > 0x7fffffffLL || sub_cap < 32 || sub_cap > kSegSubMax) return cudaErrorInvalidValue;
  const size_t smem = (size_t)pow2_at_least(sub_cap) * sizeof(uint32_t);
  static cudaError_t st = cudaSuccess;
  static bool set = false;
  MM_TRY_CUDA(smem_limit_once(k_seg_build, kSegBuildSmemMax, st, set));
  k_seg_build<<<(unsigned)n_groups, kWinThreads, smem, s>>>(groups, block_off, slot, ang2, sub_cap, ent, ent_ang,
                                                           kept);
  return cudaGetLastError();
}

// One CTA per group and column.  Per sub-window: the sub-window's u into shared memory (one
// coalesced pass over its chunks), then each thread reduces kSegRange consecutive sorted entries:
// it sums (u, cos 2psi u, sin 2psi u) in registers along each run of equal slots and adds a run's
// sums to the group's per-slot totals once, with a shared-memory atomic for the first and last run
// of its range (which other threads may share) and a plain update for the runs between them (which
// lie wholly in its range).  Last, one float4 global atomic per distinct pixel of the group.
__global__ void __launch_bounds__(kWinThreads, 2) k_point_seg32(
    const PGroup* __restrict__ groups, const int64_t* __restrict__ block_off, const uint32_t* __restrict__ ent,
    const float* __restrict__ ent_ang, const int32_t* __restrict__ kept, const int32_t* __restrict__ slot_pix,
    int sub_cap, const float* __restrict__ u, int64_t u_stride, int nrhs, const int32_t* __restrict__ done,
    int done_stride, float4* __restrict__ y4, int64_t y_stride4, PtMaps maps) {
  extern __shared__ __align__(16) float smem_f[];
  float* acc = smem_f;                   // [3][kAccStride]
  float* us = smem_f + 3 * kAccStride;   // [sub_cap] u of the sub-window, sample l at us[l]
  const PGroup G = groups[blockIdx.x];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int ls = seg_log_s(G.n_blk, G.log_w, sub_cap);
  const int n_sub = 1 << (G.log_w - ls);
  const int64_t stride = seg_stride(G.n_blk, ls);
  PGroup S = G;   // the current sub-window as a group of window 2^log_s
  S.log_w = ls;
  const ChunkWalk cw = chunk_walk(S.log_w, lane);
  const int n_pad = acc_index(G.n_slots);
  y4 = group_map(y4, nrhs * y_stride4, maps);
  for (int r = 0; r < nrhs; r++) {
    if (done != nullptr && done[(int64_t)r * done_stride] != 0) continue;
    const float* ur = u + r * u_stride;
    for (int k = threadIdx.x; k < n_pad; k += kWinThreads) {
      acc[k] = 0.f;
      acc[kAccStride + k] = 0.f;
      acc[2 * kAccStride + k] = 0.f;
    }
    for (int sw = 0; sw < n_sub; sw++) {
      S.w0 = G.w0 + ((int64_t)sw << ls);
      const int nk = __ldg(kept + G.sub0 + sw);
      const int64_t base = G.ent_off + (int64_t)sw * stride;
      const int n_rng = (nk + kSegRange - 1) / kSegRange;
      // this thread's first range, loaded before the staging pass so both latencies overlap
      uint4 pe[kSegRange / 4];
      float4 pa[kSegRange / 4];
      if ((int)threadIdx.x < n_rng) {
        const uint4* ep = reinterpret_cast<const uint4*>(ent + base + (int64_t)threadIdx.x * kSegRange);
        const float4* ap = reinterpret_cast<const float4*>(ent_ang + base + (int64_t)threadIdx.x * kSegRange);
#pragma unroll
        for (int v = 0; v < kSegRange / 4; v++) {
          pe[v] = __ldcs(ep + v);
          pa[v] = __ldcs(ap + v);
        }
      }
      __syncthreads();   // the previous sub-window's u is no longer read (and the sums are cleared)
      for (int c0 = warp * cw.cpi; c0 < S.n_blk; c0 += kWarps * cw.cpi) {
        const int c = c0 + cw.sub;
        if (c >= S.n_blk) continue;
        int64_t lo;
        int len;
        group_chunk(S, block_off, c, lo, len);
        const int l0 = c << ls;
        visit_unit(
            S, block_off, c, S.log_w, cw,
            [&](int64_t a0, int q) {
              const int64_t i = a0 + 4 * (int64_t)q;
              const float4 v = __ldcs(reinterpret_cast<const float4*>(ur + i));
              const int l = l0 + (int)(i - lo);
              us[l] = v.x;
              us[l + 1] = v.y;
              us[l + 2] = v.z;
              us[l + 3] = v.w;
            },
            [&](int64_t i) { us[l0 + (int)(i - lo)] = __ldcs(ur + i); });
      }
      __syncthreads();
      for (int g = threadIdx.x; g < n_rng; g += kWinThreads) {
        if (g != (int)threadIdx.x) {
          const uint4* ep = reinterpret_cast<const uint4*>(ent + base + (int64_t)g * kSegRange);
          const float4* ap = reinterpret_cast<const float4*>(ent_ang + base + (int64_t)g * kSegRange);
#pragma unroll
          for (int v = 0; v < kSegRange / 4; v++) {
            pe[v] = __ldcs(ep + v);
            pa[v] = __ldcs(ap + v);
          }
        }
        uint32_t cur = pe[0].x >> 16;
        float s0 = 0.f, s1 = 0.f, s2 = 0.f;
        bool first = true;
        auto flush = [&](bool shared_run) {
          if (cur == kNoSlot) return;
          const int k = acc_index((int)cur);
          if (shared_run) {
            atomicAdd(acc + k, s0);
            atomicAdd(acc + kAccStride + k, s1);
            atomicAdd(acc + 2 * kAccStride + k, s2);
          } else {
            acc[k] += s0;
            acc[kAccStride + k] += s1;
            acc[2 * kAccStride + k] += s2;
          }
        };
#pragma unroll
        for (int i = 0; i < kSegRange; i++) {
          const uint4& e4 = pe[i / 4];
          const float4& a4 = pa[i / 4];
          const uint32_t e = (i % 4 == 0) ? e4.x : (i % 4 == 1) ? e4.y : (i % 4 == 2) ? e4.z : e4.w;
          const float ang = (i % 4 == 0) ? a4.x : (i % 4 == 1) ? a4.y : (i % 4 == 2) ? a4.z : a4.w;
          const uint32_t sl = e >> 16;
          if (sl != cur) {
            flush(first);
            first = false;
            cur = sl;
            s0 = s1 = s2 = 0.f;
          }
          if (sl != kNoSlot) {
            float cs, sn;
            weights_of_angle(ang, cs, sn);
            const float y = us[e & 0xFFFFu];
            s0 += y;
            s1 = fmaf(cs, y, s1);
            s2 = fmaf(sn, y, s2);
          }
        }
        flush(true);
      }
    }
    __syncthreads();
    float4* yr = y4 + r * y_stride4;
    for (int k = threadIdx.x; k < G.n_slots; k += kWinThreads) {
      const int32_t p = __ldg(slot_pix + G.slot_off + k);
      const int j = acc_index(k);
      atomicAdd(yr + p, make_float4(acc[j], acc[kAccStride + j], acc[2 * kAccStride + j], 0.f));
    }
    __syncthreads();   // the next column clears the sums
  }
}

cudaError_t launch_point_seg32(const PGroup* groups, int64_t n_groups, const int64_t* block_off,
                               const uint32_t* ent, const float* ent_ang, const int32_t* kept,
                               const int32_t* slot_pix, int sub_cap, const float* u, int64_t u_stride,
                               int nrhs, const int32_t* done, int done_stride, float* y4, int64_t y_stride,
                               const PtMaps& maps, cudaStream_t s) {
  if (n_groups == 0 || nrhs <= 0) return cudaSuccess;
  if (n_groups > 0x7fffffffLL || u_stride % 4 != 0 || sub_cap < 32 || sub_cap > kSegSubMax)
    return cudaErrorInvalidValue;
  const size_t smem = (size_t)3 * kAccStride * sizeof(float) + (size_t)sub_cap * sizeof(float);
  static cudaError_t st = cudaSuccess;
  static bool set = false;
  MM_TRY_CUDA(smem_limit_once(k_point_seg32, kPointSegSmemMax, st, set));
  k_point_seg32<<<(unsigned)n_groups, kWinThreads, smem, s>>>(groups, block_off, ent, ent_ang, kept, slot_pix,
                                                               sub_cap, u, u_stride, nrhs, done, done_stride,
                                                               reinterpret_cast<float4*>(y4), y_stride / 4, maps);
  return cudaGetLastError();
}

// ---- FP32 right-hand side input: t = G d rounded to FP32 (0 at flagged and excised samples) ----
template <typename D>
__global__ void k_d_to_t32(const int32_t* __restrict__ lpix, const D* __restrict__ d, int64_t N, int64_t d_stride,
                           float* __restrict__ t, int64_t t_stride) {
  const D* dr = d + blockIdx.y * d_stride;
  float* tr = t + blockIdx.y * t_stride;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < N; i += (int64_t)gridDim.x * blockDim.x)
    __stcs(tr + i, (__ldg(lpix + i) >= 0) ? (float)__ldcs(dr + i) : 0.f);
}

cudaError_t launch_d_to_t32(const int32_t* lpix, const void* d, int d_is_fp32, int64_t N, int nrhs, float* t,
                            int64_t t_stride, cudaStream_t s) {
  if (N == 0 || nrhs <= 0) return cudaSuccess;
  const int64_t g = std::min<int64_t>((N + 255) / 256, 16 * (int64_t)sm_count());
  const dim3 grid((unsigned)g, nrhs);
  if (d_is_fp32)
    k_d_to_t32<float><<<grid, 256, 0, s>>>(lpix, reinterpret_cast<const float*>(d), N, N, t, t_stride);
  else
    k_d_to_t32<double><<<grid, 256, 0, s>>>(lpix, reinterpret_cast<const double*>(d), N, N, t, t_stride);
  return cudaGetLastError();
}

// ---- the FP64-class (double-float) P^T over the windows ------------------------------------------
// Each group's sums are 64-bit fixed-point integers in shared memory: integer shared-memory
// atomics are native, and integer sums do not depend on the order of the additions.  The column's
// u values are bounded by umax (the df64 N^-1 tiles record max |u|), the weights by 1 and a slot
// receives at most 2^15 samples, so with 2^k, k = 45 - floor(log2 umax), a slot's sum stays below
// 2^61 while one unit is about 2^-46 umax, under the double-float operator's own relative error.

// round(f 2^k) as a 64-bit integer with integer instructions only (the FP32 -> 64-bit conversion
// instruction runs on the FP64 pipe); zero and subnormal f give 0
__device__ __forceinline__ long long fixed_of(float f, int k) {
  const uint32_t b = __float_as_uint(f);
  const int e = (int)((b >> 23) & 0xffu);
  if (e == 0) return 0;
  const long long m = (long long)((b & 0x7fffffu) | 0x800000u);
  const int sh = e - 150 + k;
  long long v;
  if (sh >= 0) v = m << min(sh, 39);
  else if (sh > -40) v = (m + (1ll << (-sh - 1))) >> (-sh);
  else v = 0;
  return (b >> 31) ? -v : v;
}
__device__ __forceinline__ long long fixed_of(df v, int k) { return fixed_of(v.hi, k) + fixed_of(v.lo, k); }

// round(f 2^(32 + e)) with sc = 2^e (a normal float) and |f sc| < 2^30, rounding the magnitude:
// x = |f| sc (exact), its integer part and its fraction (x - floor(x), exact for x >= 0) times 2^32
// as two 32-bit conversions, then the sign.
__device__ __forceinline__ long long fixed_fast(float f, float sc) {
  const float x = fabsf(f) * sc;
  const float h = floorf(x);
  const unsigned long long m =
      ((unsigned long long)__float2uint_rn(h) << 32) + __float2uint_rn((x - h) * 4294967296.f);
  return f < 0.f ? -(long long)m : (long long)m;
}
__device__ __forceinline__ long long fixed_fast(df v, float sc) { return fixed_fast(v.hi, sc) + fixed_fast(v.lo, sc); }

constexpr size_t kPointDfSmem = (size_t)3 * kAccStride * sizeof(unsigned long long);

__global__ void __launch_bounds__(kWinThreads, 2) k_point_win_df(
    const PGroup* __restrict__ groups, const int64_t* __restrict__ block_off,
    const uint16_t* __restrict__ slot, const int32_t* __restrict__ slot_pix, const float4* __restrict__ wdf,
    const float2* __restrict__ u, int64_t u_stride, const uint32_t* __restrict__ amax, int nrhs,
    const int32_t* __restrict__ done, int done_stride, double* __restrict__ y4, int64_t y_stride) {
  extern __shared__ unsigned long long acc64[];   // [3][kAccStride]
  const PGroup G = groups[blockIdx.x];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, warps = blockDim.x >> 5;
  const int n_pad = acc_index(G.n_slots);
  for (int r = 0; r < nrhs; r++) {
    if (done != nullptr && done[(int64_t)r * done_stride] != 0) continue;
    const uint32_t ub = __ldg(amax + r);
    if (ub == 0u) continue;   // u = 0: nothing to add
    double* yr = y4 + r * y_stride;
    if (ub >= 0x7f800000u) {   // a non-finite u: poison the outputs so the solver sees it
      for (int k = threadIdx.x; k < G.n_slots; k += blockDim.x)
        atomicAdd(yr + 4 * (int64_t)__ldg(slot_pix + G.slot_off + k), __longlong_as_double(0x7ff8000000000000ll));
      continue;
    }
    const int e_u = (int)((ub >> 23) & 0xffu) - 127;   // umax in [2^e_u, 2^(e_u + 1)) (subnormal: e_u = -127)
    const int ks = 45 - e_u;
    // sums in units of 2^-ks: |y| < 2^(e_u + 1) gives |y 2^(ks - 32)| < 2^14; the fast conversion
    // takes the scale 2^(ks - 32) as a normal float (all but umax below 2^-114)
    const bool fast = ks - 32 <= 126;
    const float sc = fast ? __int_as_float((ks - 32 + 127) << 23) : 0.f;
    const double unit = __longlong_as_double((long long)(1023 - ks) << 52);   // 2^-ks
    const float2* ur = u + r * u_stride;
    for (int k = threadIdx.x; k < n_pad; k += blockDim.x) {
      acc64[k] = 0ull;
      acc64[kAccStride + k] = 0ull;
      acc64[2 * kAccStride + k] = 0ull;
    }
    __syncthreads();
    auto add = [&](uint32_t sl, float4 w, float2 y2) {
      if (sl == kNoSlot) return;
      const df y = df_make(y2.x, y2.y);
      const df cy = df_make(w.x, w.y) * y, sy = df_make(w.z, w.w) * y;
      const int k = acc_index((int)sl);
      if (fast) {
        atomicAdd(acc64 + k, (unsigned long long)fixed_fast(y, sc));
        atomicAdd(acc64 + kAccStride + k, (unsigned long long)fixed_fast(cy, sc));
        atomicAdd(acc64 + 2 * kAccStride + k, (unsigned long long)fixed_fast(sy, sc));
      } else {
        atomicAdd(acc64 + k, (unsigned long long)fixed_of(y, ks));
        atomicAdd(acc64 + kAccStride + k, (unsigned long long)fixed_of(cy, ks));
        atomicAdd(acc64 + 2 * kAccStride + k, (unsigned long long)fixed_of(sy, ks));
      }
    };
    // a warp takes 128 samples of a row at a time (32 when the rows are that short), lane = sample: every
    // load is one contiguous piece, and the next piece's are in flight while this one is added (four
    // consecutive samples per lane: 350 us for 25M samples, now 202; 26 B per sample)
    constexpr int U = 2;
    struct Piece {
      uint16_t s[U];
      float4 w[U];
      float2 y[U];
    };
    const int lp = min(G.log_w, 6), lsp = G.log_w - lp, n_pc = G.n_blk << lsp;   // pieces of 2^lp <= 32 U samples
    auto load = [&](int c, Piece& q) {
      int64_t lo = 0;
      int len = 0;
      if (c < n_pc) group_unit(G, block_off, c, lp, lo, len);
#pragma unroll
      for (int j = 0; j < U; j++) {
        const int o = 32 * j + lane;
        q.s[j] = o < len ? __ldcs(slot + lo + o) : kNoSlot;
        if (o < len) {
          q.w[j] = __ldcs(wdf + lo + o);
          q.y[j] = __ldcs(ur + lo + o);
        }
      }
    };
    // warps take contiguous ranges of the pieces, so warps running at the same time sit far apart on the
    // focal plane and rarely add to the same pixel at once
    const int per = (n_pc + warps - 1) / warps, c_end = min(n_pc, (warp + 1) * per);
    Piece cur, nxt;
    load(warp * per < c_end ? warp * per : n_pc, cur);
    for (int c = warp * per; c < c_end; c++) {
      load(c + 1 < c_end ? c + 1 : n_pc, nxt);
#pragma unroll
      for (int j = 0; j < U; j++) add(cur.s[j], cur.w[j], cur.y[j]);
      cur = nxt;
    }
    __syncthreads();
    for (int k = threadIdx.x; k < G.n_slots; k += blockDim.x) {
      const int64_t p = __ldg(slot_pix + G.slot_off + k);
      const int j = acc_index(k);
      atomicAdd(yr + 4 * p, (double)(long long)acc64[j] * unit);
      atomicAdd(yr + 4 * p + 1, (double)(long long)acc64[kAccStride + j] * unit);
      atomicAdd(yr + 4 * p + 2, (double)(long long)acc64[2 * kAccStride + j] * unit);
    }
    __syncthreads();   // the next column clears the sums
  }
}

cudaError_t launch_point_win_df(const PGroup* groups, int64_t n_groups, const WinSize& size, const int64_t* block_off,
                                const uint16_t* slot, const int32_t* slot_pix, const float4* wdf,
                                const float2* u, int64_t u_stride, const uint32_t* amax, int nrhs,
                                const int32_t* done, int done_stride, double* y4, int64_t y_stride,
                                cudaStream_t s) {
  if (n_groups == 0 || nrhs <= 0) return cudaSuccess;
  if (n_groups > 0x7fffffffLL || u_stride % 4 != 0 || y_stride % 4 != 0) return cudaErrorInvalidValue;
  static cudaError_t st = cudaSuccess;
  static bool set = false;
  MM_TRY_CUDA(smem_limit_once(k_point_win_df, kPointDfSmem, st, set));
  k_point_win_df<<<(unsigned)n_groups, size.threads, kPointDfSmem, s>>>(groups, block_off, slot, slot_pix, wdf, u,
                                                                         u_stride, amax, nrhs, done, done_stride, y4,
                                                                         y_stride);
  return cudaGetLastError();
}

}  // namespace mm
