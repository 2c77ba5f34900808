// Adjoint of the Lanczos sub-pixel-shift render (Section 2, Step 8 variant):
// the weights of the shift and their slopes.
//
// The Lanczos model is J = Lz_d(I_n): the model I rendered at the integer
// offset n = floor(x + 1/2) (and likewise in y), convolved periodically with
// the normalised Lanczos-3 weights w_a(d) of the fraction d = x - n.  The
// parameters other than the offset enter through I alone and the offset
// through d alone (n is piecewise constant), so for an upstream gradient g
//   dL/dtheta = <Lz^T g, dI/dtheta>          (flux, log r_e, e1, e2, Sersic n)
//   dL/dx     = <(dLz/d d_x)^T g, I>,
// and likewise dL/dy.  The adjoint kernels (render_bwd*.cu) take one forward
// transform of g for all of them: on the spectrum the transposed convolutions
// are multiplications by the conjugate responses of w and of the slopes w' =
// dw/dd, folded into the phase tables; for the real-space terms they are formed
// from the patch where it is read.  Measured
// on 10k 64 x 64 galaxies: 0.335 ms a call; a kernel that wrote the three
// convolved patches, an adjoint pass over each and a synchronisation to size
// them took 1.453 ms (the plain adjoint of one pass takes 0.24 ms).
#pragma once

#include "internal.h"

namespace mog {

// L'(t) of L(t) = sinc(t) sinc(t/3) on |t| < 3: with sinc'(t) =
// (cos(pi t) - sinc(t)) / t, L' = sinc'(t) sinc(t/3) + sinc(t) (cos(pi t/3) -
// sinc(t/3)) / t; 0 at t = 0 and for |t| >= 3.  Near 0 the difference
// cos - sinc cancels in FP32, so there the Taylor series of L about 0,
// 1 - (10/54) (pi t)^2 + (112/9720) (pi t)^4 - ..., is differentiated instead.
__device__ __forceinline__ float lanczos_tap_slope(float t) {
  const float at = fabsf(t);
  if (t == 0.0f || at >= 3.0f) return 0.0f;
  constexpr float P2 = PI_F * PI_F;
  if (at < 0.05f) return t * P2 * (-(10.0f / 27.0f) + (448.0f / 9720.0f) * P2 * t * t);
  float s1, c1, s3, c3;
  sincospif(t, &s1, &c1);
  sincospif(t * (1.0f / 3.0f), &s3, &c3);
  const float pt = PI_F * t;
  const float sinc1 = s1 / pt, sinc3 = 3.0f * s3 / pt;
  return ((c1 - sinc1) * sinc3 + sinc1 * (c3 - sinc3)) / t;
}

// Galaxy g's weights w_a = L(a - d) / S and slopes w'_a = (-L'(a - d) S +
// L(a - d) sum_b L'(b - d)) / S^2, a = -3..3, S = sum_b L(b - d), in the ADJ_LW
// layout (one warp: lanes 0-6 along x, 8-14 along y).
//
// The slopes' sum is zero, and what rounding leaves of it (9e-8 rms) would go,
// times sum(g I), into d/dx: for a wide galaxy and an upstream gradient with a
// mean that is far more than the rounding of d/dx itself.  So the stored ones
// add up to zero exactly: six of them are multiples of the last place of the
// seventh, the centre's, which is minus their sum.  (One to five galaxies, an
// upstream of N(1/4, 1): errors of d/dx and d/dy against 64 bits, over the
// gradients' norm, 1.6e-7 to 5.6e-7 without, 3e-8 to 1.4e-7 with, medians per
// side and column; the phase shift's adjoint has 4e-8 to 1.6e-7.)
__device__ __forceinline__ void lanczos_weights_and_slopes_warp(const BatchView& b, int64_t g, float* out) {
  const int lane = threadIdx.x & 31;
  const float c = (lane & 8) ? b.y[g] : b.x[g];
  const float d = c - floorf(c + 0.5f);
  const bool tap = lane < 16 && (lane & 7) < 7;
  const float t = (float)((lane & 7) - 3) - d;
  const float lv = tap ? lanczos_tap(t) : 0.0f, lp = tap ? lanczos_tap_slope(t) : 0.0f;
  float s = lv, sp = lp;
#pragma unroll
  for (int o = 1; o < 8; o <<= 1) {
    s += __shfl_xor_sync(0xffffffffu, s, o);
    sp += __shfl_xor_sync(0xffffffffu, sp, o);
  }
  const float inv = tap ? 1.0f / s : 0.0f;
  const bool centre = (lane & 7) == 3;
  const float slope = centre ? 0.0f : (lv * sp - lp * s) * inv * inv;   // |slope| < 1.4
  float rest = slope;
#pragma unroll
  for (int o = 1; o < 8; o <<= 1) rest += __shfl_xor_sync(0xffffffffu, rest, o);
  // 2^e <= |centre| < 2^(e + 1), with room for what the steps below change of it;
  // the grid is 2^(e - 23).  Down to e = -6 the sums are 32-bit integers.
  const int e = max(-6, min(0, ilogbf(fmaf(1e-5f, fabsf(rest), fabsf(rest)))));
  const int units = __float2int_rn(scalbnf(slope, 23 - e));
  int sum = units;
#pragma unroll
  for (int o = 1; o < 8; o <<= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
  if (lane < 16) {
    const int at = (lane & 8) * 2 + (lane & 7);
    out[at] = lv * inv;
    out[at + 8] = scalbnf((float)(centre ? -sum : units), e - 23);
  }
}

}  // namespace mog
