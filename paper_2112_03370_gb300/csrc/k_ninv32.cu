// FP32 block-Toeplitz product u = N^-1 t (Eq. MADCAP, stbmm of Sect. 3.1): overlap-save tiles with
// the transform held in registers.
//
// A tile of L = 2M real samples is packed as M complex values z[n] = t[2n] + i t[2n+1] and
// transformed by M = R1 R2 16 points, 32 complex values per thread (M / 32 threads):
//   P1  radix R1 over n = j + S1 i (S1 = M / R1), straight from global memory into registers;
//   P2  radix R2 inside each of the R1 sub-transforms;
//   F   the last radix 16 of two groups of 16 frequencies at a time, the group c and its mirror
//       M/16 - c: frequencies k and M - k of the real-input pair update
//       Z'[k] = a_k Z[k] + i b_k conj(Z[M-k]) then sit in one thread, which runs both radix-16
//       butterflies, the update and both inverse butterflies without touching shared memory;
//   P2', P1'  the inverse passes; P1' writes the tile's valid outputs straight to global memory.
// A warp handles the same sub-transforms (k1 and its mirror R1 - k1) in P2, F and P2', so those three
// need no CTA barrier between them: two barriers per tile, and warps on their shared-memory phases
// overlap with warps on their arithmetic.
// Shared memory only carries the four exchanges between the passes: 8 touches of every value
// instead of the 16 of in-place passes in shared memory, which were bound by the shared-memory pipe
// and instruction issue (89k warp instructions and 22.8k shared wavefronts in 40k cycles per
// 32768-sample tile; here 54k and 11.2k in 25k cycles).  What bounds it now: latency at 16 warps per
// SM between the arithmetic (FMA pipe 53% busy, its throttle the first of the stalls) and the shared-memory
// pipe (50%).
// Measured (GB300, t and u in HBM, kernel alone, before -> now): 512 blocks x 524,288 samples, lambda
// 8192: 2.18 -> 1.34 ms; 256 x 524,288, lambda 1024: 0.69 -> 0.35 ms; 64 x 262,144, lambda 2048:
// 120 -> 64 us; 4 x 65,536, lambda 1024: 28 -> 10 us (plus 4% since the rotation constants carry their low
// parts, fft_reg.cuh).
//
// Geometry by tile size: 32768 samples R1 = R2 = 32 (512 threads, one CTA per SM), 16384 samples
// 32 x 16 (256 threads, two), 8192 samples 16 x 16 (128 threads, four).
//
// Twiddles of P1: W_M^{j k} for the thread's j from w, w^2, w^3 and w^4, w^8, .. (a table per CTA)
// with at most one product; P2: a table of W_{S1}^{j2 k}.
//
// Shared layout: position p at p + p/16, so P1 and P2 (16 consecutive positions per half-warp) and F
// (lanes 17 apart) are free of bank conflicts; a thread's lane enumerates k2 of its group
// c = k1 + R1 k2, because positions of neighbouring k1 fall on one bank.
#include <cstdint>
#include <type_traits>

#include "fft_reg.cuh"
#include "mm_internal.cuh"

namespace mm {

namespace {

using namespace rfft;

template <int LOGM>
struct NGeom {
  static constexpr int M = 1 << LOGM;
  static constexpr int L = 2 * M;
  static constexpr int NT = M / 32;
  static constexpr int R1 = LOGM >= 13 ? 32 : 16;
  static constexpr int R2 = LOGM >= 14 ? 32 : 16;
  static constexpr int S1 = M / R1;
  static constexpr int B1 = 32 / R1, B2 = 32 / R2;
  static constexpr int NG = M / 16;   // groups of 16 frequencies
  static constexpr int P1 = S1 + S1 / 16;   // padded stride of the R1 sub-transforms
  static constexpr int T1ROWS = 3 + (R1 / 4 - 1);
  static constexpr int CTAS = LOGM >= 14 ? 1 : LOGM == 13 ? 2 : 4;
  static constexpr int kImage = T1ROWS * S1 + R2 * 16;   // twiddle tables of P1 and P2
  static constexpr size_t kSmem = (size_t)(M + M / 16 + kImage) * sizeof(float2);
  static_assert(R1 * R2 * 16 == M && S1 == 16 * R2, "geometry");
};

// power of w held by row r of the P1 table: 1, 2, 3, 4, 8, 12, ..
__host__ __device__ constexpr int t1_power(int r) { return r < 3 ? r + 1 : 4 * (r - 2); }

// groups of thread t: k1 and k2 of its first and second group (thread 0 holds the two groups that
// mirror onto themselves, c = 0 and c = NG / 2)
template <int R1, int R2>
__host__ __device__ __forceinline__ void thread_groups(int t, int& k1a, int& k2a, int& k1b, int& k2b) {
  const int u = t / R2, q = t % R2;
  if (u > 0) {
    k1a = u; k2a = q; k1b = R1 - u; k2b = R2 - 1 - q;
  } else if (q < R2 / 2) {
    k1a = 0; k2a = q; k1b = 0; k2b = q == 0 ? R2 / 2 : R2 - q;
  } else {
    k1a = R1 / 2; k2a = q - R2 / 2; k1b = R1 / 2; k2b = R2 - 1 - k2a;
  }
}

// a[k] *= w^k (FWD) or conj(w)^k, k < R, from the P1 table rows at column j
template <int R, bool FWD, int O, int N>
__device__ __forceinline__ void twiddle_p1(float2 (&a)[N], const float2* __restrict__ t1, int s1) {
  const float2 w1 = t1[0], w2 = t1[s1], w3 = t1[2 * s1];
  a[O + 1] = twid<FWD>(a[O + 1], w1);
  a[O + 2] = twid<FWD>(a[O + 2], w2);
  a[O + 3] = twid<FWD>(a[O + 3], w3);
#pragma unroll
  for (int b = 1; b < R / 4; b++) {
    const float2 wb = t1[(2 + b) * s1];
    a[O + 4 * b] = twid<FWD>(a[O + 4 * b], wb);
    a[O + 4 * b + 1] = twid<FWD>(a[O + 4 * b + 1], mul(wb, w1));
    a[O + 4 * b + 2] = twid<FWD>(a[O + 4 * b + 2], mul(wb, w2));
    a[O + 4 * b + 3] = twid<FWD>(a[O + 4 * b + 3], mul(wb, w3));
  }
}

// Z'[k], Z'[M - k] of one frequency pair: sc (a x + b y', a y + b x') and the mirror (b is shared).  The
// block's scale comes last: at low frequencies a and b cancel almost completely (a + b -> H(f), small for
// red noise), and scaled coefficients, each rounded on its own, are a gain error there that differs from
// block to block.  Error of u per mode below 0.005 Hz (knee 1 Hz, slope 1.5, lambda 8192, one tile emulated
// on the host): 3.1e-6 of rms u with scaled coefficients, 2.2e-6 so; map error of the FP32 right-hand side
// of the ground workload (1.07e9 samples): 6.2e-6 -> 1.7e-6.  A x of it takes 10.31 ms either way.
__device__ __forceinline__ void pair_update(float2& z, float2& zp, float a, float ap, float b, float sc) {
  const float2 o = make_float2(sc * (a * z.x + b * zp.y), sc * (a * z.y + b * zp.x));
  zp = make_float2(sc * (ap * zp.x + b * z.y), sc * (ap * zp.y + b * z.x));
  z = o;
}

__device__ __forceinline__ void prefetch_l2_input(const void* p, uint32_t bytes) {
  asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(__cvta_generic_to_global(p)), "r"(bytes)
               : "memory");
}

__device__ __forceinline__ void cp_async16(void* dst, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src)
               : "memory");
}

}  // namespace

template <int LOGM, bool MULTI>
__global__ void __launch_bounds__(NGeom<LOGM>::NT, NGeom<LOGM>::CTAS) k_ninv32(const TileArgs a_in) {
  using G = NGeom<LOGM>;
  constexpr int NT = G::NT, R1 = G::R1, R2 = G::R2, S1 = G::S1;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  float2* sm = reinterpret_cast<float2*>(smem_raw);
  float2* t1 = sm + G::M + G::M / 16;
  const float2* t2 = t1 + G::T1ROWS * S1;

  const int tid = threadIdx.x;
  const int rhs = (int)(blockIdx.x % a_in.nrhs);
  const TileDesc seg = a_in.tiles[blockIdx.x / a_in.nrhs];
  const float* x = reinterpret_cast<const float*>(a_in.x);
  float* y = reinterpret_cast<float*>(a_in.y);
  const float4* tab = reinterpret_cast<const float4*>(a_in.tab);
  const int32_t* done = a_in.done;
  if constexpr (MULTI) {   // this tile's problem
    const ProbPtrs pp = a_in.probs[seg.prob];
    x = reinterpret_cast<const float*>(pp.x);
    y = reinterpret_cast<float*>(pp.y);
    tab = reinterpret_cast<const float4*>(pp.tab);
    done = pp.done;
  }
  if (done != nullptr && done[(int64_t)rhs * a_in.done_stride] != 0) return;
  x += rhs * a_in.x_stride;
  y += rhs * a_in.y_stride;
  tab += (int64_t)seg.tab * (12 * NT) + tid;
  const float sc = (float)seg.scale;

  // twiddle tables (one contiguous image) on their way to shared memory while the first tile loads
  for (int i = tid; i < G::kImage / 2; i += NT)
    cp_async16(t1 + 2 * i, reinterpret_cast<const float4*>(a_in.tw) + i);
  asm volatile("cp.async.commit_group;" ::: "memory");
  int k1a, k2a, k1b, k2b;
  thread_groups<R1, R2>(tid, k1a, k2a, k1b, k2b);
  float2* const ga = sm + k1a * G::P1 + k2a * 17;
  float2* const gb = sm + k1b * G::P1 + k2b * 17;
  // P2: 16 lanes per sub-transform, a warp on the same sub-transforms (k1 and its mirror) as in F
  const int j2 = tid & 15;
  const int ku = tid / R2, km = ku == 0 ? R1 / 2 : R1 - ku;
  const int p2a = ((G::B2 == 1 && (tid & 16)) ? km : ku) * G::P1 + j2;
  const int p2b = km * G::P1 + j2;

  float2 v[32];
  for (int step = 0; step < seg.n_steps; step++) {
    const int64_t in0 = seg.in0 + (int64_t)step * seg.vstep;
    const int64_t out_lo = seg.out_lo + (int64_t)step * seg.vstep;
    const int64_t out_hi = min(out_lo + (int64_t)seg.vstep, seg.out_hi);

    // ---- P1: z[j + S1 i] from global memory, zero outside the block ----
    if (in0 >= seg.blk_lo && in0 + G::L <= seg.blk_hi) {
      const float2* src = reinterpret_cast<const float2*>(x + in0) + tid;   // in0 is a multiple of 4
#pragma unroll
      for (int b = 0; b < G::B1; b++)
#pragma unroll
        for (int i = 0; i < R1; i++) v[b * R1 + i] = __ldg(src + b * NT + i * S1);
    } else {
      const int lo = (int)max(seg.blk_lo - in0, (int64_t)0);
      const int hi = (int)min(seg.blk_hi - in0, (int64_t)G::L);
#pragma unroll
      for (int b = 0; b < G::B1; b++)
#pragma unroll
        for (int i = 0; i < R1; i++) {
          const int n = 2 * (tid + b * NT + i * S1);
          float2 f = make_float2(0.f, 0.f);
          if (n >= lo && n + 2 <= hi) {
            f = __ldg(reinterpret_cast<const float2*>(x + in0 + n));
          } else {
            if (n >= lo && n < hi) f.x = __ldg(x + in0 + n);
            if (n + 1 >= lo && n + 1 < hi) f.y = __ldg(x + in0 + n + 1);
          }
          v[b * R1 + i] = f;
        }
    }
    if (tid == 0 && step + 1 < seg.n_steps) {   // the next tile's new samples start on their way to L2
      int64_t lo = max(in0 + G::L, seg.blk_lo), hi = min(in0 + G::L + (int64_t)seg.vstep, seg.blk_hi);
      lo = (lo + 3) & ~(int64_t)3;   // 16-byte aligned and inside the block
      hi &= ~(int64_t)3;
      if (hi > lo) prefetch_l2_input(x + lo, (uint32_t)((hi - lo) * 4));
    }
    auto p1_fwd = [&](auto bc) {
      constexpr int b = decltype(bc)::value;
      const int j = tid + b * NT;
      float2* d = sm + j + (j >> 4);
      dft<R1, true, b * R1>(v);
      twiddle_p1<R1, true, b * R1>(v, t1 + j, S1);
#pragma unroll
      for (int k = 0; k < R1; k++) d[k * G::P1] = v[b * R1 + k];
    };
    auto p2 = [&](auto bc, auto fwd) {
      constexpr int b = decltype(bc)::value;
      constexpr bool FWD = decltype(fwd)::value;
      float2* d = sm + (b == 0 ? p2a : p2b);
#pragma unroll
      for (int i = 0; i < R2; i++) v[b * R2 + i] = d[i * 17];
      if constexpr (FWD) {
        dft<R2, true, b * R2>(v);
#pragma unroll
        for (int k = 1; k < R2; k++) v[b * R2 + k] = mul(v[b * R2 + k], t2[k * 16 + j2]);
      } else {
#pragma unroll
        for (int k = 1; k < R2; k++) v[b * R2 + k] = mulc(v[b * R2 + k], t2[k * 16 + j2]);
        dft<R2, false, b * R2>(v);
      }
#pragma unroll
      for (int k = 0; k < R2; k++) d[k * 17] = v[b * R2 + k];
    };
    auto p1_inv = [&](auto bc) {
      constexpr int b = decltype(bc)::value;
      const int j = tid + b * NT;
      const float2* d = sm + j + (j >> 4);
#pragma unroll
      for (int k = 0; k < R1; k++) v[b * R1 + k] = d[k * G::P1];
      twiddle_p1<R1, false, b * R1>(v, t1 + j, S1);
      dft<R1, false, b * R1>(v);
    };
    using I0 = std::integral_constant<int, 0>;
    using I1 = std::integral_constant<int, 1>;

    if (step == 0) {
      asm volatile("cp.async.wait_all;" ::: "memory");
      __syncthreads();
    }
    p1_fwd(I0{});
    if constexpr (G::B1 == 2) p1_fwd(I1{});
    __syncthreads();

    p2(I0{}, std::true_type{});
    if constexpr (G::B2 == 2) p2(I1{}, std::true_type{});
    // ---- F: radix 16 of both groups, pair update, inverse radix 16 ----
    float4 c0 = __ldg(tab), c1 = __ldg(tab + NT), c2 = __ldg(tab + 2 * NT);   // slots 0..3
    __syncwarp();
#pragma unroll
    for (int e = 0; e < 16; e++) {
      v[e] = ga[e];
      v[16 + e] = gb[e];
    }
    dft16<true, 0>(v);
    dft16<true, 16>(v);
#pragma unroll
    for (int h = 0; h < 4; h++) {
      const float f[12] = {c0.x, c0.y, c0.z, c0.w, c1.x, c1.y, c1.z, c1.w, c2.x, c2.y, c2.z, c2.w};
      if (h < 3) {
        c0 = __ldg(tab + (3 * h + 3) * NT);
        c1 = __ldg(tab + (3 * h + 4) * NT);
        c2 = __ldg(tab + (3 * h + 5) * NT);
      }
      if (tid != 0) {
#pragma unroll
        for (int s = 0; s < 4; s++) {
          const int e = 4 * h + s;
          pair_update(v[e], v[31 - e], f[3 * s], f[3 * s + 1], f[3 * s + 2], sc);
        }
      } else {   // the groups that mirror onto themselves
#pragma unroll
        for (int s = 0; s < 4; s++) {
          const int e = 4 * h + s;
          const float a = f[3 * s], ap = f[3 * s + 1], b = f[3 * s + 2];
          if (e < 7) {
            pair_update(v[e + 1], v[15 - e], a, ap, b, sc);
          } else if (e < 15) {
            pair_update(v[16 + e - 7], v[31 - (e - 7)], a, ap, b, sc);
          } else {   // k = 0: (a, b) = (f0, f1); k = M/2: b = 0, a = f2
            v[0] = make_float2(sc * (a * v[0].x + ap * v[0].y), sc * (a * v[0].y + ap * v[0].x));
            v[8] = make_float2(sc * (b * v[8].x), sc * (b * v[8].y));
          }
        }
      }
    }
    dft16<false, 0>(v);
    dft16<false, 16>(v);
#pragma unroll
    for (int e = 0; e < 16; e++) {
      ga[e] = v[e];
      gb[e] = v[16 + e];
    }
    __syncwarp();

    p2(I0{}, std::false_type{});
    if constexpr (G::B2 == 2) p2(I1{}, std::false_type{});
    __syncthreads();

    p1_inv(I0{});
    if constexpr (G::B1 == 2) p1_inv(I1{});
    // the tile's valid outputs; the next tile's P1 writes only the column this thread has read
    const int lo = (int)(out_lo - in0), hi = (int)(out_hi - in0);
    float* yo = y + in0;
#pragma unroll
    for (int b = 0; b < G::B1; b++)
#pragma unroll
      for (int i = 0; i < R1; i++) {
        const int n = 2 * (tid + b * NT + i * S1);
        const float2 f = v[b * R1 + i];
        if (n >= lo && n + 2 <= hi) {
          __stcs(reinterpret_cast<float2*>(yo + n), f);
        } else {
          if (n >= lo && n < hi) yo[n] = f.x;
          if (n + 1 >= lo && n + 1 < hi) yo[n + 1] = f.y;
        }
      }
  }
}

// Pair table of k_ninv32: thread t, slot e: (a_k, a_{M-k}, b_k) of the pair that slot holds, in the
// order the kernel reads them (12 float4 per thread, [12][NT] per table).  H [n_tab][kM + 1] is the
// 2 kM-point circulant spectrum; a shorter tile samples the same symbol more coarsely.
template <int LOGM>
__global__ void k_pair_table_reg(const double* __restrict__ H, const double* __restrict__ costab, int32_t n_tab,
                                 float* __restrict__ out) {
  using G = NGeom<LOGM>;
  constexpr int kStep = kM / G::M;
  const int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (idx >= (int64_t)n_tab * G::NT * 16) return;
  const int tabi = (int)(idx / (G::NT * 16));
  const int t = (int)(idx / 16) % G::NT, e = (int)(idx % 16);
  const double* h = H + (int64_t)tabi * (kM + 1);
  auto coef = [&](int k, double& av, double& bv) {
    const double hk = h[k * kStep], hm = h[(G::M - k) * kStep];
    const double S = 0.5 * (hk + hm), D = 0.5 * (hk - hm);
    const double cth = costab[k * kStep];
    const double sth = costab[(k * kStep - kL / 4) & (kL - 1)];
    av = (S - D * sth) / (double)G::M;
    bv = D * cth / (double)G::M;
  };
  int k1a, k2a, k1b, k2b;
  thread_groups<G::R1, G::R2>(t, k1a, k2a, k1b, k2b);
  const int ca = k1a + G::R1 * k2a, cb = k1b + G::R1 * k2b;
  double f0, f1, f2, tmp;
  if (t != 0 || e < 15) {
    const int k = t != 0 ? ca + G::NG * e : e < 7 ? G::NG * (e + 1) : cb + G::NG * (e - 7);
    coef(k, f0, f2);
    coef(G::M - k, f1, tmp);
  } else {
    coef(0, f0, f1);
    coef(G::M / 2, f2, tmp);
  }
  const float f[3] = {(float)f0, (float)f1, (float)f2};
  for (int c = 0; c < 3; c++) {
    const int i = 3 * e + c;   // float i of the thread's 48
    out[((int64_t)tabi * 12 + i / 4) * G::NT * 4 + t * 4 + i % 4] = f[c];
  }
}

// twiddle image of k_ninv32 from tw[k] = W_kM^k: P1 rows [T1ROWS][S1], then P2 [R2][16]
template <int LOGM>
__global__ void k_twiddle_image(const float2* __restrict__ tw, float2* __restrict__ out) {
  using G = NGeom<LOGM>;
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= G::kImage) return;
  const int r = i - G::T1ROWS * G::S1;
  out[i] = r < 0 ? tw[t1_power(i / G::S1) * (i % G::S1) * (kM / G::M)] : tw[(r / 16) * (r % 16) * (kM / G::S1)];
}
size_t twiddle_image_len(int logm) {
  return logm == 14 ? NGeom<14>::kImage : logm == 13 ? NGeom<13>::kImage : NGeom<12>::kImage;
}
cudaError_t launch_twiddle_image(int logm, const float2* tw, float2* out, cudaStream_t s) {
  const unsigned nb = (unsigned)((twiddle_image_len(logm) + 255) / 256);
  if (logm == 14) k_twiddle_image<14><<<nb, 256, 0, s>>>(tw, out);
  else if (logm == 13) k_twiddle_image<13><<<nb, 256, 0, s>>>(tw, out);
  else if (logm == 12) k_twiddle_image<12><<<nb, 256, 0, s>>>(tw, out);
  else return cudaErrorInvalidValue;
  return cudaGetLastError();
}

cudaError_t launch_pair_table_reg(int logm, const double* H, int32_t n_tab, const double* costab, float* out,
                                  cudaStream_t s) {
  if (n_tab == 0) return cudaSuccess;
  const int64_t n = (int64_t)n_tab << (logm - 1);   // 16 slots x M / 32 threads
  const unsigned nb = (unsigned)((n + 255) / 256);
  if (logm == 14) k_pair_table_reg<14><<<nb, 256, 0, s>>>(H, costab, n_tab, out);
  else if (logm == 13) k_pair_table_reg<13><<<nb, 256, 0, s>>>(H, costab, n_tab, out);
  else if (logm == 12) k_pair_table_reg<12><<<nb, 256, 0, s>>>(H, costab, n_tab, out);
  else return cudaErrorInvalidValue;
  return cudaGetLastError();
}
size_t pair_table_reg_floats(int logm, int32_t n_tab) { return (size_t)n_tab * 48 << (logm - 5); }

int ninv32_init() {
  static const cudaError_t e = [] {
    cudaError_t r = cudaSuccess;
    auto set = [&](auto k, size_t b) {
      if (r == cudaSuccess) r = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)b);
    };
    set(k_ninv32<14, false>, NGeom<14>::kSmem);
    set(k_ninv32<14, true>, NGeom<14>::kSmem);
    set(k_ninv32<13, false>, NGeom<13>::kSmem);
    set(k_ninv32<13, true>, NGeom<13>::kSmem);
    set(k_ninv32<12, false>, NGeom<12>::kSmem);
    set(k_ninv32<12, true>, NGeom<12>::kSmem);
    return r;
  }();
  return e == cudaSuccess ? MM_OK : cuda_fail(e, "FP32 Toeplitz tile attributes");
}

template <int LOGM, bool MULTI>
static cudaError_t launch_one(const TileArgs& a, cudaStream_t s) {
  const int64_t n = a.n_tiles * a.nrhs;
  if (n == 0) return cudaSuccess;
  if (n > 0x7fffffffLL) return cudaErrorInvalidConfiguration;
  k_ninv32<LOGM, MULTI><<<(unsigned)n, NGeom<LOGM>::NT, NGeom<LOGM>::kSmem, s>>>(a);
  return cudaGetLastError();
}

// u = N^-1 t on tiles of 2^(logm + 1) samples: t, u [nrhs][stride] (strides multiples of 4), a.tab from
// launch_pair_table_reg, a.tw from launch_twiddle_image; a.probs set: tiles of several problems (nrhs 1)
cudaError_t launch_ninv32(int logm, const TileArgs& a, cudaStream_t s) {
  if (a.x_stride % 4 != 0 || a.y_stride % 4 != 0) return cudaErrorInvalidValue;
  if (a.probs != nullptr) {
    if (a.nrhs != 1) return cudaErrorInvalidValue;
    if (logm == 14) return launch_one<14, true>(a, s);
    if (logm == 13) return launch_one<13, true>(a, s);
    if (logm == 12) return launch_one<12, true>(a, s);
    return cudaErrorInvalidValue;
  }
  if (logm == 14) return launch_one<14, false>(a, s);
  if (logm == 13) return launch_one<13, false>(a, s);
  if (logm == 12) return launch_one<12, false>(a, s);
  return cudaErrorInvalidValue;
}

}  // namespace mm
