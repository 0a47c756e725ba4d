// Block conjugate gradients on s right-hand sides (Algorithm 2 in its block Orthomin form with
// R_0 = [b_1 .. b_s]): tall-skinny block products and the small dense steps.
//
// Layouts: a block of t pixel-domain vectors is [t][n][4] (IQU + pad per pixel, pad = 0).
// Search blocks (Z, A Z, P, A P, M R) are float32; X, R and every t x t matrix are float64.
// Tall-skinny products run on the FP32 units (GB300's FP64 rate is 1/64 of FP32) with FP64
// accumulation across CTAs; the solver's accuracy is restored by FP64 residual checks.
#include "df64.cuh"
#include "mm_block.cuh"
#include "mm_internal.cuh"

namespace mm {

namespace {
constexpr int kNT = 256;
}  // namespace

// Partial Gram products: out_part[blk][i tb + j] = sum over this CTA's contiguous range of pixels
// of <A_i, B_j> (3 components), FP32 products and sums, FP64 per-CTA totals.  ta, tb <= kMaxBlk.
// A is a float4 block, B a float4 or float64 block (R); columns selected through idx_a / idx_b
// (identity when null).

// The same partial Gram products for small blocks (ta <= MA, tb <= MB): every thread streams its
// pixels (grid-stride, coalesced) and keeps the ta tb dot products in registers; then a block
// reduction in FP64.  (The staged kernel below keeps most threads idle when t is small.)
template <typename TB, int MA, int MB>
__global__ void __launch_bounds__(kNT) k_bgram_small(const float4* __restrict__ A, int ta,
                                                      const int* __restrict__ idx_a,
                                                      const TB* __restrict__ B, int tb,
                                                      const int* __restrict__ idx_b, int64_t n,
                                                      double* __restrict__ out_part) {
  __shared__ double red[kNT / 32][MA * MB];
  float acc[MA][MB];
#pragma unroll
  for (int i = 0; i < MA; i++)
#pragma unroll
    for (int j = 0; j < MB; j++) acc[i][j] = 0.f;
  for (int64_t p = (int64_t)blockIdx.x * kNT + threadIdx.x; p < n; p += (int64_t)gridDim.x * kNT) {
    float bx[MB], by[MB], bz[MB];
#pragma unroll
    for (int j = 0; j < MB; j++) {
      bx[j] = by[j] = bz[j] = 0.f;
      if (j < tb) {
        const int64_t col = idx_b ? idx_b[j] : j;
        if constexpr (sizeof(TB) == sizeof(float4)) {
          const float4 v = __ldg(reinterpret_cast<const float4*>(B) + col * n + p);
          bx[j] = v.x; by[j] = v.y; bz[j] = v.z;
        } else {
          const double* v = reinterpret_cast<const double*>(B) + 4 * (col * n + p);
          bx[j] = (float)v[0]; by[j] = (float)v[1]; bz[j] = (float)v[2];
        }
      }
    }
#pragma unroll
    for (int i = 0; i < MA; i++) {
      if (i < ta) {
        const float4 a = __ldg(A + (int64_t)(idx_a ? idx_a[i] : i) * n + p);
#pragma unroll
        for (int j = 0; j < MB; j++) acc[i][j] += a.x * bx[j] + a.y * by[j] + a.z * bz[j];
      }
    }
  }
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
#pragma unroll
  for (int i = 0; i < MA; i++)
#pragma unroll
    for (int j = 0; j < MB; j++) {
      double v = (double)acc[i][j];
      for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
      if (lane == 0) red[warp][i * MB + j] = v;
    }
  __syncthreads();
  if (threadIdx.x < MA * MB) {
    const int i = threadIdx.x / MB, j = threadIdx.x % MB;
    if (i < ta && j < tb) {
      double v = 0.0;
      for (int w = 0; w < kNT / 32; w++) v += red[w][threadIdx.x];
      out_part[(int64_t)blockIdx.x * kMaxBlk * kMaxBlk + i * tb + j] = v;
    }
  }
}

template <int MA, int MB>
static void bgram_small(const float* A, int ta, const int* idx_a, const void* B, int b_is_fp64, int tb,
                        const int* idx_b, int64_t n, double* part, int nblk, cudaStream_t s) {
  if (b_is_fp64)
    k_bgram_small<double4_16a, MA, MB><<<nblk, kNT, 0, s>>>(reinterpret_cast<const float4*>(A), ta, idx_a,
                                                            reinterpret_cast<const double4_16a*>(B), tb, idx_b, n,
                                                            part);
  else
    k_bgram_small<float4, MA, MB><<<nblk, kNT, 0, s>>>(reinterpret_cast<const float4*>(A), ta, idx_a,
                                                       reinterpret_cast<const float4*>(B), tb, idx_b, n, part);
}

// The same partial Gram products for wide blocks, NC = 16, 32 or 64 columns on each side: each thread a
// 4 x 4 tile of (i, j) in registers, (NC / 4)^2 threads for all pairs and 256 / that many groups of threads on
// different pixels; kGR 64 / NC pixels of both blocks staged per step as [pixel][component][column] (rows
// padded to keep 16-byte alignment and spread the staging stores over banks), so a thread's four a values
// and four b values of one pixel component are two 16-byte shared loads for 16 FMAs.  The groups' totals
// meet in FP64 at the end.  With 64-column tiles for 16 columns 240 of the 256 threads multiplied zeros and
// added them in FP64: 65,536 pixels, 16 x 16 columns 88 -> 42 us.
constexpr int kGR = 24;   // 2 x 19.6 KB of static shared memory
template <typename TB, int NC>
__global__ void __launch_bounds__(kNT) k_bgram_tiled(const float4* __restrict__ A, int ta,
                                                      const int* __restrict__ idx_a,
                                                      const TB* __restrict__ B, int tb,
                                                      const int* __restrict__ idx_b, int64_t n,
                                                      double* __restrict__ out_part) {
  static_assert(kNT == 256 && kMaxBlk == 64 && (NC == 16 || NC == 32 || NC == 64), "256 threads of 4 x 4 pairs");
  constexpr int kTiles = NC / 4, kGroups = kNT / (kTiles * kTiles), kPix = kGR * 64 / NC, kRow = NC + 4;
  constexpr int kHalf = kPix * 3 * kRow;
  static_assert(2 * kHalf * 4 >= NC * NC * 8, "the totals reuse the staging buffers");
  __shared__ __align__(16) float smem[2 * kHalf];
  float(*sa)[3][kRow] = reinterpret_cast<float(*)[3][kRow]>(smem);
  float(*sb)[3][kRow] = reinterpret_cast<float(*)[3][kRow]>(smem + kHalf);
  const int grp = threadIdx.x / (kTiles * kTiles), in = threadIdx.x % (kTiles * kTiles);
  const int ti = in / kTiles, tj = in % kTiles;
  double tot[4][4];   // FP64 totals of the per-chunk FP32 sums (two-level summation)
#pragma unroll
  for (int u = 0; u < 4; u++)
#pragma unroll
    for (int v = 0; v < 4; v++) tot[u][v] = 0.0;
  const int64_t per = (n + gridDim.x - 1) / gridDim.x;
  const int64_t p0 = (int64_t)blockIdx.x * per, p1 = min(n, p0 + per);
  for (int64_t base = p0; base < p1; base += kPix) {
    const int cnt = (int)min((int64_t)kPix, p1 - base);
    // staging: consecutive threads take consecutive pixels of one column (coalesced loads)
    for (int e = threadIdx.x; e < kPix * NC; e += kNT) {
      const int r = e % kPix, i = e / kPix;
      float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
      if (r < cnt && i < ta) v = __ldg(A + (int64_t)(idx_a ? idx_a[i] : i) * n + base + r);
      sa[r][0][i] = v.x; sa[r][1][i] = v.y; sa[r][2][i] = v.z;
      float x = 0.f, y = 0.f, z = 0.f;
      if (r < cnt && i < tb) {
        const int64_t col = idx_b ? idx_b[i] : i;
        if constexpr (sizeof(TB) == sizeof(float4)) {
          const float4 w = __ldg(reinterpret_cast<const float4*>(B) + col * n + base + r);
          x = w.x; y = w.y; z = w.z;
        } else {
          const double2* w = reinterpret_cast<const double2*>(B) + 2 * (col * n + base + r);
          const double2 xy = w[0];
          x = (float)xy.x; y = (float)xy.y; z = (float)w[1].x;
        }
      }
      sb[r][0][i] = x; sb[r][1][i] = y; sb[r][2][i] = z;
    }
    __syncthreads();
    float acc[4][4];
#pragma unroll
    for (int u = 0; u < 4; u++)
#pragma unroll
      for (int v = 0; v < 4; v++) acc[u][v] = 0.f;
    for (int r = grp; r < cnt; r += kGroups) {
#pragma unroll
      for (int c = 0; c < 3; c++) {
        const float4 a = *reinterpret_cast<const float4*>(&sa[r][c][4 * ti]);
        const float4 b = *reinterpret_cast<const float4*>(&sb[r][c][4 * tj]);
        const float av[4] = {a.x, a.y, a.z, a.w}, bv[4] = {b.x, b.y, b.z, b.w};
#pragma unroll
        for (int u = 0; u < 4; u++)
#pragma unroll
          for (int v = 0; v < 4; v++) acc[u][v] = fmaf(av[u], bv[v], acc[u][v]);
      }
    }
#pragma unroll
    for (int u = 0; u < 4; u++)
#pragma unroll
      for (int v = 0; v < 4; v++) tot[u][v] += f32_to_f64_bits(acc[u][v]);
    __syncthreads();
  }
  double* o = out_part + (int64_t)blockIdx.x * kMaxBlk * kMaxBlk;
  if constexpr (kGroups > 1) {   // the groups add their totals one after the other (a fixed order)
    double* sum = reinterpret_cast<double*>(smem);   // [NC][NC]
    for (int g = 0; g < kGroups; g++) {
      if (grp == g)
#pragma unroll
        for (int u = 0; u < 4; u++)
#pragma unroll
          for (int v = 0; v < 4; v++) {
            double* q = sum + (4 * ti + u) * NC + 4 * tj + v;
            *q = g == 0 ? tot[u][v] : *q + tot[u][v];
          }
      __syncthreads();
    }
    for (int e = threadIdx.x; e < ta * tb; e += kNT) o[e] = sum[(e / tb) * NC + e % tb];
  } else {
#pragma unroll
    for (int u = 0; u < 4; u++)
#pragma unroll
      for (int v = 0; v < 4; v++) {
        const int i = 4 * ti + u, j = 4 * tj + v;
        if (i < ta && j < tb) o[i * tb + j] = tot[u][v];
      }
  }
}

template <int NC>
static void bgram_tiled(const float* A, int ta, const int* idx_a, const void* B, int b_is_fp64, int tb,
                        const int* idx_b, int64_t n, double* part, int nblk, cudaStream_t s) {
  if (b_is_fp64)
    k_bgram_tiled<double4_16a, NC><<<nblk, kNT, 0, s>>>(reinterpret_cast<const float4*>(A), ta, idx_a,
                                                        reinterpret_cast<const double4_16a*>(B), tb, idx_b, n, part);
  else
    k_bgram_tiled<float4, NC><<<nblk, kNT, 0, s>>>(reinterpret_cast<const float4*>(A), ta, idx_a,
                                                   reinterpret_cast<const float4*>(B), tb, idx_b, n, part);
}

// G[i][j] = sum over CTAs of out_part (fixed order: deterministic)
// One warp per output: lane l sums partials l, l + 32, ... in order, then a fixed shuffle tree
// (deterministic, and 32 loads in flight instead of one serial chain over all CTAs).
__device__ __forceinline__ double warp_sum_strided(const double* __restrict__ part, int64_t stride, int nblk) {
  const int lane = threadIdx.x & 31;
  double s = 0.0;
  for (int b = lane; b < nblk; b += 32) s += part[(int64_t)b * stride];
  for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  return s;
}

__global__ void k_bgram_reduce(const double* __restrict__ part, int nblk, int npair,
                               double* __restrict__ G) {
  const int pr = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  if (pr >= npair) return;
  const double s = warp_sum_strided(part + pr, (int64_t)kMaxBlk * kMaxBlk, nblk);
  if ((threadIdx.x & 31) == 0) G[pr] = s;
}

cudaError_t launch_bgram(const float* A, int ta, const int* idx_a, const void* B, int b_is_fp64,
                         int tb, const int* idx_b, int64_t n, double* part, int nblk, double* G,
                         cudaStream_t s) {
  if (ta <= 0 || tb <= 0) return cudaSuccess;
  if (ta > kMaxBlk || tb > kMaxBlk) return cudaErrorInvalidValue;
  if (ta <= 4 && tb <= 4) {
    bgram_small<4, 4>(A, ta, idx_a, B, b_is_fp64, tb, idx_b, n, part, nblk, s);
  } else if (ta == 1 && tb <= 16) {
    bgram_small<1, 16>(A, ta, idx_a, B, b_is_fp64, tb, idx_b, n, part, nblk, s);
  } else if (ta <= 16 && tb <= 16) {
    bgram_tiled<16>(A, ta, idx_a, B, b_is_fp64, tb, idx_b, n, part, nblk, s);
  } else if (ta <= 32 && tb <= 32) {
    bgram_tiled<32>(A, ta, idx_a, B, b_is_fp64, tb, idx_b, n, part, nblk, s);
  } else {
    bgram_tiled<64>(A, ta, idx_a, B, b_is_fp64, tb, idx_b, n, part, nblk, s);
  }
  k_bgram_reduce<<<(ta * tb + 7) / 8, 256, 0, s>>>(part, nblk, ta * tb, G);
  return cudaGetLastError();
}

// out_j (+)= sign * sum_i A_i C[i][j] for j < v (A: float32 [t][n]; C: FP64 [t][v] row-major with
// leading dimension ldc; out: FP64 or FP32 block, column j stored at idx_out[j] (or j)).  mode 0:
// out = sign * sum, mode 1: out += sign * sum.  A CTA stages kCP pixels of every input column and
// the coefficients in shared memory, then each thread forms 8 output columns of one pixel (warp w
// takes columns 8 w .. 8 w + 7, its lanes consecutive pixels, so the stores coalesce and each
// warp owns its columns' norm partials).  With norm_part != null (FP64 outputs), per-CTA partials
// of ||out_j||^2 are written.
constexpr int kCP = 32;
template <typename TO>
__global__ void __launch_bounds__(kNT) k_bcombine(TO* __restrict__ out, const int* __restrict__ idx_out,
                                                   int v, const float4* __restrict__ A, int t,
                                                   const double* __restrict__ C, int ldc, double sign,
                                                   int mode, int64_t n, double* __restrict__ norm_part) {
  static_assert(kNT == 256 && kMaxBlk == 64 && kCP == 32, "8 warps x 8 columns, 32 pixels per step");
  __shared__ __align__(16) float4 sA[kMaxBlk][kCP];     // 32 KB
  __shared__ __align__(16) float cs[kMaxBlk][kMaxBlk];  // 16 KB
  for (int e = threadIdx.x; e < t * v; e += kNT) cs[e / v][e % v] = (float)(sign * C[(e / v) * ldc + (e % v)]);
  const int r = threadIdx.x & 31, g = threadIdx.x >> 5;   // pixel in the chunk, column group
  const int j0 = 8 * g;
  const int nj = max(0, min(8, v - j0));
  double nrm[8];
#pragma unroll
  for (int jj = 0; jj < 8; jj++) nrm[jj] = 0.0;
  const int64_t n_chunks = (n + kCP - 1) / kCP;
  for (int64_t ch = blockIdx.x; ch < n_chunks; ch += gridDim.x) {
    const int64_t base = ch * kCP;
    const int cnt = (int)min((int64_t)kCP, n - base);
    __syncthreads();   // the previous chunk is no longer read (and the coefficients are staged)
    for (int e = threadIdx.x; e < t * kCP; e += kNT) {
      const int i = e / kCP, q = e % kCP;
      sA[i][q] = (q < cnt) ? __ldg(A + (int64_t)i * n + base + q) : make_float4(0.f, 0.f, 0.f, 0.f);
    }
    __syncthreads();
    if (nj == 0 || r >= cnt) continue;
    float ax[8], ay[8], az[8];
#pragma unroll
    for (int jj = 0; jj < 8; jj++) ax[jj] = ay[jj] = az[jj] = 0.f;
    for (int i = 0; i < t; i++) {
      const float4 a = sA[i][r];
      const float4 c0 = *reinterpret_cast<const float4*>(&cs[i][j0]);
      const float4 c1 = *reinterpret_cast<const float4*>(&cs[i][j0 + 4]);
      const float c[8] = {c0.x, c0.y, c0.z, c0.w, c1.x, c1.y, c1.z, c1.w};
#pragma unroll
      for (int jj = 0; jj < 8; jj++) {
        ax[jj] = fmaf(a.x, c[jj], ax[jj]);
        ay[jj] = fmaf(a.y, c[jj], ay[jj]);
        az[jj] = fmaf(a.z, c[jj], az[jj]);
      }
    }
    const int64_t p = base + r;
#pragma unroll
    for (int jj = 0; jj < 8; jj++) {
      if (jj >= nj) break;
      const int64_t col = idx_out ? idx_out[j0 + jj] : (j0 + jj);
      if constexpr (sizeof(TO) == sizeof(float4)) {
        float4* o = reinterpret_cast<float4*>(out) + col * n + p;
        float4 cur = mode ? *o : make_float4(0.f, 0.f, 0.f, 0.f);
        cur.x += ax[jj]; cur.y += ay[jj]; cur.z += az[jj];
        cur.w = 0.f;
        *o = cur;
      } else {
        double* o = reinterpret_cast<double*>(out) + 4 * (col * n + p);
        double x0 = mode ? o[0] : 0.0, x1 = mode ? o[1] : 0.0, x2 = mode ? o[2] : 0.0;
        x0 += f32_to_f64_bits(ax[jj]); x1 += f32_to_f64_bits(ay[jj]); x2 += f32_to_f64_bits(az[jj]);
        o[0] = x0; o[1] = x1; o[2] = x2; o[3] = 0.0;
        if (norm_part) nrm[jj] += x0 * x0 + x1 * x1 + x2 * x2;
      }
    }
  }
  if (norm_part) {
#pragma unroll
    for (int jj = 0; jj < 8; jj++) {
      double v2 = nrm[jj];
      for (int o = 16; o > 0; o >>= 1) v2 += __shfl_xor_sync(0xffffffffu, v2, o);
      if (r == 0 && jj < nj) norm_part[(int64_t)(j0 + jj) * gridDim.x + blockIdx.x] = v2;
    }
  }
}

// Narrow blocks (v, t <= kCombJ): each thread streams pixels (grid-stride) and forms all v outputs
// of its pixel in registers; no staging, so a column or two costs one pass over A.
constexpr int kCombJ = 16;
// columns whose loads are in flight together: FP32 outputs 4 (65,536 pixels, 16 x 16: 18.8 -> 11.5 us: one column's
// load at a time, and each output read after the last one's store, waited for memory); FP64 outputs 1 (30 us, with
// 4 columns' 32-byte pixels in registers 35)
template <typename TO>
constexpr int kCombU = sizeof(TO) == sizeof(float4) ? 4 : 1;
__device__ __forceinline__ float4 load_pixel(const float4* o) { return *o; }
__device__ __forceinline__ void store_pixel(float4* o, float4 v) { *o = v; }
// 16-byte accesses to the pixel's 32 bytes
__device__ __forceinline__ double4_16a load_pixel(const double4_16a* o) {
  const double2 a = reinterpret_cast<const double2*>(o)[0], b = reinterpret_cast<const double2*>(o)[1];
  return double4_16a{a.x, a.y, b.x, b.y};
}
__device__ __forceinline__ void store_pixel(double4_16a* o, double4_16a v) {
  reinterpret_cast<double2*>(o)[0] = make_double2(v.x, v.y);
  reinterpret_cast<double2*>(o)[1] = make_double2(v.z, v.w);
}
template <typename TO, int J>
__global__ void __launch_bounds__(kNT) k_bcombine_stream(TO* __restrict__ out, const int* __restrict__ idx_out,
                                                   int v, const float4* __restrict__ A, int t,
                                                   const double* __restrict__ C, int ldc, double sign,
                                                   int mode, int64_t n, double* __restrict__ norm_part) {
  __shared__ float cs[kMaxBlk * kMaxBlk];
  __shared__ double red[J][kNT / 32];
  constexpr int kU = kCombU<TO>;
  for (int e = threadIdx.x; e < t * v; e += kNT) cs[e] = (float)(sign * C[(e / v) * ldc + (e % v)]);
  __syncthreads();
  for (int j0 = 0; j0 < v; j0 += J) {
    const int nj = min(J, v - j0);
    double nrm[J];
#pragma unroll
    for (int jj = 0; jj < J; jj++) nrm[jj] = 0.0;
    for (int64_t p = (int64_t)blockIdx.x * kNT + threadIdx.x; p < n; p += (int64_t)gridDim.x * kNT) {
      float ax[J], ay[J], az[J];
#pragma unroll
      for (int jj = 0; jj < J; jj++) ax[jj] = ay[jj] = az[jj] = 0.f;
      for (int i0 = 0; i0 < t; i0 += kU) {
        float4 a[kU];
#pragma unroll
        for (int u = 0; u < kU; u++)
          a[u] = i0 + u < t ? __ldg(A + (int64_t)(i0 + u) * n + p) : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
        for (int u = 0; u < kU; u++) {
          if (i0 + u >= t) break;
#pragma unroll
          for (int jj = 0; jj < J; jj++) {
            const float c = (jj < nj) ? cs[(i0 + u) * v + j0 + jj] : 0.f;
            ax[jj] = fmaf(a[u].x, c, ax[jj]);
            ay[jj] = fmaf(a[u].y, c, ay[jj]);
            az[jj] = fmaf(a[u].z, c, az[jj]);
          }
        }
      }
#pragma unroll
      for (int j1 = 0; j1 < J; j1 += kU) {
        TO cur[kU];   // kU columns' pixels before the first of them is stored
        int64_t at[kU];
#pragma unroll
        for (int u = 0; u < kU; u++) {
          if (j1 + u < nj) {
            at[u] = (idx_out ? idx_out[j0 + j1 + u] : (j0 + j1 + u)) * n + p;
            if (mode) cur[u] = load_pixel(out + at[u]);
            else cur[u] = TO{};
          }
        }
#pragma unroll
        for (int u = 0; u < kU; u++) {
          const int jj = j1 + u;
          if (jj >= nj) break;
          if constexpr (sizeof(TO) == sizeof(float4)) {
            cur[u].x += ax[jj]; cur[u].y += ay[jj]; cur[u].z += az[jj];
          } else {
            cur[u].x += f32_to_f64_bits(ax[jj]); cur[u].y += f32_to_f64_bits(ay[jj]); cur[u].z += f32_to_f64_bits(az[jj]);
            if (norm_part) nrm[jj] += cur[u].x * cur[u].x + cur[u].y * cur[u].y + cur[u].z * cur[u].z;
          }
          cur[u].w = 0;
          store_pixel(out + at[u], cur[u]);
        }
      }
    }
    if (norm_part) {
      // a warp reduces its J values together, exchanging halves, then the warps' sums in order
      const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
      int o = 16;
#pragma unroll
      for (int h = J / 2; h > 0; h >>= 1, o >>= 1) {
        const bool up = (lane & o) != 0;
#pragma unroll
        for (int j = 0; j < h; j++) {
          const double give = up ? nrm[j] : nrm[j + h], keep = up ? nrm[j + h] : nrm[j];
          nrm[j] = keep + __shfl_xor_sync(0xffffffffu, give, o);
        }
      }
      for (; o > 0; o >>= 1) nrm[0] += __shfl_xor_sync(0xffffffffu, nrm[0], o);
      if (lane % (32 / J) == 0) red[lane / (32 / J)][warp] = nrm[0];
      __syncthreads();
      if (threadIdx.x < nj) {
        double acc = 0.0;
#pragma unroll
        for (int w = 0; w < kNT / 32; w++) acc += red[threadIdx.x][w];
        norm_part[(int64_t)(j0 + threadIdx.x) * gridDim.x + blockIdx.x] = acc;
      }
      __syncthreads();
    }
  }
}

__global__ void k_norm_reduce(const double* __restrict__ part, int nblk, int v, double* __restrict__ out) {
  const int j = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  if (j >= v) return;
  const double s = warp_sum_strided(part + (int64_t)j * nblk, 1, nblk);
  if ((threadIdx.x & 31) == 0) out[j] = s;
}

cudaError_t launch_bcombine(void* out, int out_is_fp64, const int* idx_out, int v, const float* A, int t,
                            const double* C, int ldc, double sign, int mode, int64_t n, double* norm_part,
                            int nblk, double* norms, cudaStream_t s) {
  if (v <= 0) return cudaSuccess;
  if (t > kMaxBlk || v > kMaxBlk) return cudaErrorInvalidValue;
  const bool narrow = v <= kCombJ && t <= kCombJ;
  if (out_is_fp64) {
    if (narrow && v <= 4)   // few outputs: fewer registers, more resident warps
      k_bcombine_stream<double4_16a, 4><<<nblk, kNT, 0, s>>>(reinterpret_cast<double4_16a*>(out), idx_out, v,
                                                             reinterpret_cast<const float4*>(A), t, C, ldc, sign,
                                                             mode, n, norm_part);
    else if (narrow)
      k_bcombine_stream<double4_16a, kCombJ><<<nblk, kNT, 0, s>>>(reinterpret_cast<double4_16a*>(out), idx_out, v,
                                                                  reinterpret_cast<const float4*>(A), t, C, ldc,
                                                                  sign, mode, n, norm_part);
    else
      k_bcombine<double4_16a><<<nblk, kNT, 0, s>>>(reinterpret_cast<double4_16a*>(out), idx_out, v,
                                                   reinterpret_cast<const float4*>(A), t, C, ldc, sign, mode,
                                                   n, norm_part);
  } else {
    if (narrow && v <= 4)
      k_bcombine_stream<float4, 4><<<nblk, kNT, 0, s>>>(reinterpret_cast<float4*>(out), idx_out, v,
                                                        reinterpret_cast<const float4*>(A), t, C, ldc, sign, mode, n,
                                                        nullptr);
    else if (narrow)
      k_bcombine_stream<float4, kCombJ><<<nblk, kNT, 0, s>>>(reinterpret_cast<float4*>(out), idx_out, v,
                                                             reinterpret_cast<const float4*>(A), t, C, ldc, sign, mode,
                                                             n, nullptr);
    else
      k_bcombine<float4><<<nblk, kNT, 0, s>>>(reinterpret_cast<float4*>(out), idx_out, v,
                                              reinterpret_cast<const float4*>(A), t, C, ldc, sign, mode, n,
                                              nullptr);
  }
  if (norm_part && out_is_fp64) k_norm_reduce<<<(v + 7) / 8, 256, 0, s>>>(norm_part, nblk, v, norms);
  return cudaGetLastError();
}

// W_j = M_BD R_{idx_j} in FP32 (j < v; idx null = identity); R float64 [.][n][4] or float4
template <typename TR>
__global__ void k_bprecond(const double* __restrict__ minv, const TR* __restrict__ R,
                           const int* __restrict__ idx, int v, int64_t n, float4* __restrict__ W) {
  const int64_t tot = (int64_t)v * n;
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < tot; e += (int64_t)gridDim.x * blockDim.x) {
    const int j = (int)(e / n);
    const int64_t p = e - (int64_t)j * n;
    const int64_t o = (int64_t)(idx ? idx[j] : j) * n + p;
    double r0, r1, r2;
    if constexpr (sizeof(TR) == sizeof(float4)) {
      const float4 f = R[o];
      r0 = f.x; r1 = f.y; r2 = f.z;
    } else {
      const double* r = reinterpret_cast<const double*>(R) + 4 * o;
      r0 = r[0]; r1 = r[1]; r2 = r[2];
    }
    const double* m = minv + 6 * p;
    const double z0 = m[0] * r0 + m[1] * r1 + m[2] * r2;
    const double z1 = m[1] * r0 + m[3] * r1 + m[4] * r2;
    const double z2 = m[2] * r0 + m[4] * r1 + m[5] * r2;
    W[e] = make_float4((float)z0, (float)z1, (float)z2, 0.f);
  }
}

static unsigned precond_grid(int64_t tot) {
  int64_t g = (tot + 255) / 256;
  if (g > 32 * sm_count()) g = 32 * sm_count();
  return (unsigned)g;
}

cudaError_t launch_bprecond(const double* minv, const double* R, const int* idx, int v, int64_t n,
                            float* W, cudaStream_t s) {
  if (v <= 0) return cudaSuccess;
  k_bprecond<double><<<precond_grid((int64_t)v * n), 256, 0, s>>>(minv, R, idx, v, n, reinterpret_cast<float4*>(W));
  return cudaGetLastError();
}

cudaError_t launch_bprecond32(const double* minv, const float* R, int v, int64_t n, float* W, cudaStream_t s) {
  if (v <= 0) return cudaSuccess;
  k_bprecond<float4><<<precond_grid((int64_t)v * n), 256, 0, s>>>(
      minv, reinterpret_cast<const float4*>(R), nullptr, v, n, reinterpret_cast<float4*>(W));
  return cudaGetLastError();
}

// Enlarged CG (Sect. 3.2, ECG): the split of one residual r [n][4] into t columns over contiguous
// ranges of pixels (column i keeps the pixels p with floor(p t / n) = i, zero elsewhere).
__global__ void k_bsplit(const double* __restrict__ r, int t, int64_t n, double* __restrict__ R) {
  const int64_t tot = (int64_t)t * n;
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < tot; e += (int64_t)gridDim.x * blockDim.x) {
    const int i = (int)(e / n);
    const int64_t p = e - (int64_t)i * n;
    const bool own = (p * t) / n == i;
    const double2* src = reinterpret_cast<const double2*>(r + 4 * p);
    double2* dst = reinterpret_cast<double2*>(R + 4 * e);
    dst[0] = own ? src[0] : make_double2(0.0, 0.0);
    dst[1] = own ? make_double2(src[1].x, 0.0) : make_double2(0.0, 0.0);
  }
}

cudaError_t launch_bsplit(const double* r4, int t, int64_t n, double* R, cudaStream_t s) {
  if (t <= 0 || n <= 0) return cudaSuccess;
  k_bsplit<<<precond_grid((int64_t)t * n), 256, 0, s>>>(r4, t, n, R);
  return cudaGetLastError();
}

// s_p = sum_i X_i[p] over the t columns of a FP64 block; out (+)= s when out != null, and per-CTA
// partials of ||s||^2 (norm of the summed residual of ECG, or of x = X 1).
__global__ void k_bsum(const double* __restrict__ X, int t, int64_t n, double* __restrict__ out, int accumulate,
                       double* __restrict__ norm_part) {
  __shared__ double red[kNT];
  double nrm = 0.0;
  for (int64_t p = (int64_t)blockIdx.x * kNT + threadIdx.x; p < n; p += (int64_t)gridDim.x * kNT) {
    double s0 = 0.0, s1 = 0.0, s2 = 0.0;
    for (int i = 0; i < t; i++) {
      const double* x = X + 4 * ((int64_t)i * n + p);
      s0 += x[0]; s1 += x[1]; s2 += x[2];
    }
    if (out) {
      double* o = out + 4 * p;
      if (accumulate) { s0 += o[0]; s1 += o[1]; s2 += o[2]; }
      o[0] = s0; o[1] = s1; o[2] = s2; o[3] = 0.0;
    }
    nrm += s0 * s0 + s1 * s1 + s2 * s2;
  }
  red[threadIdx.x] = nrm;
  __syncthreads();
  for (int sh = kNT / 2; sh > 0; sh >>= 1) {
    if (threadIdx.x < sh) red[threadIdx.x] += red[threadIdx.x + sh];
    __syncthreads();
  }
  if (threadIdx.x == 0) norm_part[blockIdx.x] = red[0];
}

cudaError_t launch_bsum(const double* X, int t, int64_t n, double* out, int accumulate, double* norm_part,
                        int nblk, double* norm, cudaStream_t s) {
  if (t <= 0 || t > kMaxBlk) return cudaErrorInvalidValue;
  k_bsum<<<nblk, kNT, 0, s>>>(X, t, n, out, accumulate, norm_part);
  k_norm_reduce<<<1, 32, 0, s>>>(norm_part, nblk, 1, norm);
  return cudaGetLastError();
}

// Small dense step of one iteration, one CTA, FP64:
//   G (t x t, symmetrised) = L L^T by a pivoted Cholesky with relative tolerance rank_tol;
//   Linv = L^-1 (rank x rank, lower); piv[0..rank) = pivoted columns; *rank_out = rank.
// The caller forms P = Linv Z[piv] and A P = Linv (A Z)[piv] (rows are block columns).
// Right-looking: the remaining matrix is updated after every column (each element sees the subtractions
// in the same order as a left-looking factorisation), elements and inverse columns over the threads, the
// pivot by one warp.  Bound by the latency of its t steps (a division, a square root, three barriers).
// One thread took 224 us at t = 16; now 48 us.
constexpr int kCholNT = 256;
__global__ void __launch_bounds__(kCholNT) k_bchol(const double* __restrict__ G, int t, double rank_tol,
                                                    double* __restrict__ Linv_out, int* __restrict__ piv_out,
                                                    int* __restrict__ rank_out) {
  extern __shared__ double dsm[];      // g [kMaxBlk * kLd] (the factor in its lower part), then L^-1
  constexpr int kLd = kMaxBlk + 1;
  double* g = dsm;
  double* inv = dsm + kMaxBlk * kLd;
  __shared__ int piv[kMaxBlk];
  __shared__ int s_best;
  __shared__ double s_bd, s_scale;
  const int tid = threadIdx.x, lane = tid & 31;
  for (int e = tid; e < t * t; e += kCholNT) {
    const int i = e / t, j = e % t;
    g[i * kLd + j] = 0.5 * (G[i * t + j] + G[j * t + i]);
  }
  for (int i = tid; i < t; i += kCholNT) piv[i] = i;
  __syncthreads();
  if (tid < 32) {
    double mx = 0.0;
    for (int i = lane; i < t; i += 32) mx = fmax(mx, fabs(g[i * kLd + i]));
    for (int o = 16; o > 0; o >>= 1) mx = fmax(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    if (lane == 0) s_scale = mx > 0.0 ? mx : 1e-300;
  }
  __syncthreads();
  int r = t;
  for (int k = 0; k < t; k++) {
    if (tid < 32) {   // the largest remaining diagonal, the first of equal ones
      double bd = -1.0;
      int best = k;
      for (int i = k + lane; i < t; i += 32) {
        const double d = g[i * kLd + i];
        if (d > bd) {
          bd = d;
          best = i;
        }
      }
      for (int o = 16; o > 0; o >>= 1) {
        const double d = __shfl_xor_sync(0xffffffffu, bd, o);
        const int i = __shfl_xor_sync(0xffffffffu, best, o);
        if (d > bd || (d == bd && i < best)) {
          bd = d;
          best = i;
        }
      }
      if (lane == 0) {
        s_bd = bd;
        s_best = best;
      }
    }
    __syncthreads();
    const double bd = s_bd;
    const int best = s_best;
    if (!(bd > rank_tol * s_scale)) {
      r = k;
      break;
    }
    if (best != k) {   // symmetric swap of rows and columns k and best of the remaining matrix, rows of the factor
      for (int j = tid; j < t; j += kCholNT) {
        const double tmp = g[k * kLd + j];
        g[k * kLd + j] = g[best * kLd + j];
        g[best * kLd + j] = tmp;
      }
      if (tid == 0) {
        const int tp = piv[k];
        piv[k] = piv[best];
        piv[best] = tp;
      }
      __syncthreads();
      for (int j = k + tid; j < t; j += kCholNT) {
        const double tmp = g[j * kLd + k];
        g[j * kLd + k] = g[j * kLd + best];
        g[j * kLd + best] = tmp;
      }
      __syncthreads();
    }
    const double lkk = sqrt(bd);
    for (int i = k + 1 + tid; i < t; i += kCholNT) g[i * kLd + k] = g[i * kLd + k] / lkk;
    __syncthreads();
    if (tid == 0) g[k * kLd + k] = lkk;
    const int m = t - k - 1;   // both triangles are updated: the swaps move either
    for (int e = tid; e < m * m; e += kCholNT) {
      const int i = k + 1 + e / m, j = k + 1 + e % m;
      g[i * kLd + j] -= g[i * kLd + k] * g[j * kLd + k];
    }
    __syncthreads();
  }
  // L^-1 (r x r, lower) by forward substitution, a column per thread
  for (int e = tid; e < kMaxBlk * kLd; e += kCholNT) inv[e] = 0.0;
  __syncthreads();
  for (int c = tid; c < r; c += kCholNT) {
    for (int i = c; i < r; i++) {
      double sacc = (i == c) ? 1.0 : 0.0;
      for (int m = c; m < i; m++) sacc -= g[i * kLd + m] * inv[m * kLd + c];
      inv[i * kLd + c] = sacc / g[i * kLd + i];
    }
  }
  __syncthreads();
  for (int e = tid; e < kMaxBlk * kMaxBlk; e += kCholNT) Linv_out[e] = inv[(e / kMaxBlk) * kLd + e % kMaxBlk];
  for (int i = tid; i < t; i += kCholNT) piv_out[i] = piv[i];
  if (tid == 0) *rank_out = r;
}

cudaError_t launch_bchol(const double* G, int t, double rank_tol, double* Linv, int* piv, int* rank,
                         cudaStream_t s) {
  if (t > kMaxBlk) return cudaErrorInvalidValue;
  constexpr size_t smem = 2 * kMaxBlk * (kMaxBlk + 1) * sizeof(double);
  static const cudaError_t attr =
      cudaFuncSetAttribute(k_bchol, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (attr != cudaSuccess) return attr;
  k_bchol<<<1, kCholNT, smem, s>>>(G, t, rank_tol, Linv, piv, rank);
  return cudaGetLastError();
}

// Linv as a [t][t] coefficient matrix for the combine kernel: Cmb[k][i] = Linv[i][pos(k)] where
// block column k = piv[pos]; rows/cols beyond the rank are zero.  out_i = sum_k Z_k Cmb[k][i].
__global__ void k_linv_coef(const double* __restrict__ Linv, const int* __restrict__ piv,
                            const int* __restrict__ rank, int t, double* __restrict__ Cmb) {
  const int r = *rank;
  for (int e = threadIdx.x; e < t * t; e += blockDim.x) {
    const int k = e / t, i = e % t;
    double c = 0.0;
    if (i < r) {
      for (int pos = 0; pos < r; pos++)
        if (piv[pos] == k) c = Linv[i * kMaxBlk + pos];
    }
    Cmb[k * t + i] = c;
  }
}

cudaError_t launch_linv_coef(const double* Linv, const int* piv, const int* rank, int t, double* Cmb,
                             cudaStream_t s) {
  k_linv_coef<<<1, 256, 0, s>>>(Linv, piv, rank, t, Cmb);
  return cudaGetLastError();
}

// R_j = B_j - AX_j (FP64) and norms_part of ||R_j||^2 (j < v); grid (nblk, v)
__global__ void k_bresid(const double* __restrict__ B, const double* __restrict__ AX, int64_t n,
                         double* __restrict__ R, double* __restrict__ norm_part) {
  __shared__ double red[kNT];
  const int j = blockIdx.y;
  double nrm = 0.0;
  for (int64_t p = (int64_t)blockIdx.x * kNT + threadIdx.x; p < n; p += (int64_t)gridDim.x * kNT) {
    const int64_t o = 4 * ((int64_t)j * n + p);
    const double r0 = B[o] - AX[o], r1 = B[o + 1] - AX[o + 1], r2 = B[o + 2] - AX[o + 2];
    R[o] = r0; R[o + 1] = r1; R[o + 2] = r2; R[o + 3] = 0.0;
    nrm += r0 * r0 + r1 * r1 + r2 * r2;
  }
  red[threadIdx.x] = nrm;
  __syncthreads();
  for (int sh = kNT / 2; sh > 0; sh >>= 1) {
    if (threadIdx.x < sh) red[threadIdx.x] += red[threadIdx.x + sh];
    __syncthreads();
  }
  if (threadIdx.x == 0) norm_part[(int64_t)j * gridDim.x + blockIdx.x] = red[0];
}

cudaError_t launch_bresid(const double* B, const double* AX, int v, int64_t n, double* R,
                          double* norm_part, int nblk, double* norms, cudaStream_t s) {
  if (v <= 0) return cudaSuccess;
  k_bresid<<<dim3(nblk, v), kNT, 0, s>>>(B, AX, n, R, norm_part);
  k_norm_reduce<<<(v + 7) / 8, 256, 0, s>>>(norm_part, nblk, v, norms);
  return cudaGetLastError();
}

}  // namespace mm
