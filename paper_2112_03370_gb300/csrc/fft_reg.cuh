// Register-resident complex FP32 butterflies (radix 16 and 32) of the FP32 block-Toeplitz tiles.
//
// A complex value is a float2 in one aligned register pair, so a complex sum or difference is one
// packed instruction (add/sub.rn.f32x2).  On GB300 packed FP32 issues at half the rate of scalar
// FP32, i.e. the same number of lane operations per clock (measured, 152 SMs at 2.07 GHz: fma
// 57 packed against 97 scalar lane instructions per clock and SM, add 59 against 105), so packing
// costs no arithmetic throughput and frees issue slots for the shared-memory exchanges between
// the passes.  Products and rotations by -i / +i stay scalar: packing those needs register moves.
#pragma once

#include <cuda_runtime.h>

namespace mm {
namespace rfft {

__device__ __forceinline__ float2 add2(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float2 sub2(float2 a, float2 b) {
  return __ffma2_rn(b, make_float2(-1.f, -1.f), a);   // a - b, rounded once
}
__device__ __forceinline__ float2 mul(float2 a, float2 b) {
  return make_float2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
}
// a * conj(b)
__device__ __forceinline__ float2 mulc(float2 a, float2 b) {
  return make_float2(a.x * b.x + a.y * b.y, a.y * b.x - a.x * b.y);
}
// a * w (FWD) or a * conj(w)
template <bool FWD>
__device__ __forceinline__ float2 twid(float2 a, float2 w) { return FWD ? mul(a, w) : mulc(a, w); }

// cos(2 pi e / 32), e = 0 .. 8
__device__ __forceinline__ constexpr double cos32q(int e) {
  switch (e) {
    case 0: return 1.0;
    case 1: return 0.98078528040323044913;
    case 2: return 0.92387953251128675613;
    case 3: return 0.83146961230254523708;
    case 4: return 0.70710678118654752440;
    case 5: return 0.55557023301960222474;
    case 6: return 0.38268343236508977173;
    case 7: return 0.19509032201612826785;
    default: return 0.0;
  }
}
__device__ __forceinline__ constexpr double cos32(int e) {
  e &= 31;
  if (e > 16) e = 32 - e;
  return e <= 8 ? cos32q(e) : -cos32q(16 - e);
}
__device__ __forceinline__ constexpr double sin32(int e) { return cos32(e - 8); }

// a * exp(-2 pi i e / 32) (FWD) or a * exp(+2 pi i e / 32); e is a constant after unrolling
// The same rounded constant multiplies every value of a pass in both directions, so its rounding is a gain error
// of a frequency that no averaging removes: where it is not at 45 degrees, the constant's low part goes into the
// innermost FMA.  A x of 33.6M samples at lambda 8192 against double-float, random / smooth / constant maps: 1.43, 1.84,
// 1.99e-7 (with plain constants 1.94, 2.57, 2.83e-7; low parts at 45 degrees too: 1.29, 1.61, 1.76e-7); N^-1 at lambda
// 8192 takes 4% longer (all angles: 9%).
template <bool FWD>
__device__ __forceinline__ float2 rot32(float2 a, int e) {
  e &= 31;
  if (e == 0) return a;
  if (e == 16) return make_float2(-a.x, -a.y);
  if (e == 8) return FWD ? make_float2(a.y, -a.x) : make_float2(-a.y, a.x);
  if (e == 24) return FWD ? make_float2(-a.y, a.x) : make_float2(a.y, -a.x);
  const double c = cos32(e), g = FWD ? -sin32(e) : sin32(e);
  const float ch = (float)c, sh = (float)g;
  if (e % 4 == 0) return mul(a, make_float2(ch, sh));
  const float cl = (float)(c - (double)ch), sl = (float)(g - (double)sh);
  return make_float2(fmaf(a.x, ch, fmaf(-a.y, sh, fmaf(a.x, cl, -a.y * sl))),
                     fmaf(a.x, sh, fmaf(a.y, ch, fmaf(a.x, sl, a.y * cl))));
}

template <bool FWD>
__device__ __forceinline__ void dft4(float2& a0, float2& a1, float2& a2, float2& a3) {
  const float2 s02 = add2(a0, a2), d02 = sub2(a0, a2), s13 = add2(a1, a3), d13 = sub2(a1, a3);
  a0 = add2(s02, s13);
  a2 = sub2(s02, s13);
  const float2 p = make_float2(d02.x + d13.y, d02.y - d13.x);   // d02 - i d13
  const float2 m = make_float2(d02.x - d13.y, d02.y + d13.x);   // d02 + i d13
  a1 = FWD ? p : m;
  a3 = FWD ? m : p;
}

// 16-point DFT of a[O + m], natural order in and out (y_k = sum_m a_m w^{km})
template <bool FWD, int O, int N>
__device__ __forceinline__ void dft16(float2 (&a)[N]) {
  // m = 4 m1 + m0, k = k0 + 4 k1
#pragma unroll
  for (int m0 = 0; m0 < 4; m0++) dft4<FWD>(a[O + m0], a[O + 4 + m0], a[O + 8 + m0], a[O + 12 + m0]);
#pragma unroll
  for (int k0 = 1; k0 < 4; k0++)
#pragma unroll
    for (int m0 = 1; m0 < 4; m0++) a[O + 4 * k0 + m0] = rot32<FWD>(a[O + 4 * k0 + m0], 2 * m0 * k0);
#pragma unroll
  for (int k0 = 0; k0 < 4; k0++) dft4<FWD>(a[O + 4 * k0], a[O + 4 * k0 + 1], a[O + 4 * k0 + 2], a[O + 4 * k0 + 3]);
  // y_{k0 + 4 k1} is at 4 k0 + k1: transpose (register names only)
#pragma unroll
  for (int i = 0; i < 4; i++)
#pragma unroll
    for (int j = i + 1; j < 4; j++) {
      const float2 t = a[O + 4 * i + j];
      a[O + 4 * i + j] = a[O + 4 * j + i];
      a[O + 4 * j + i] = t;
    }
}

// R-point DFT of a[O .. O + R), natural order in and out
template <int R, bool FWD, int O, int N>
__device__ __forceinline__ void dft(float2 (&a)[N]) {
  if constexpr (R == 16) {
    dft16<FWD, O>(a);
  } else {
    static_assert(R == 32 && N == 32 && O == 0, "radix");
#pragma unroll
    for (int i = 0; i < 16; i++) {   // even outputs from the sums, odd ones from the rotated differences
      const float2 s = add2(a[i], a[i + 16]), d = sub2(a[i], a[i + 16]);
      a[i] = s;
      a[i + 16] = rot32<FWD>(d, i);
    }
    dft16<FWD, 0>(a);
    dft16<FWD, 16>(a);
    float2 b[32];
#pragma unroll
    for (int i = 0; i < 16; i++) {
      b[2 * i] = a[i];
      b[2 * i + 1] = a[i + 16];
    }
#pragma unroll
    for (int i = 0; i < 32; i++) a[i] = b[i];
  }
}

}  // namespace rfft
}  // namespace mm
