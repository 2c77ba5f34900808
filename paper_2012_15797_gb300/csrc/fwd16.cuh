// Forward-render helpers of the kernels with 16 values per thread.
#pragma once

#include "fft16.cuh"
#include "internal.h"

namespace mog {

// One real-space term (its fields as in RealTermsN) added to 8 consecutive
// pixels x0.. of two rows, o[u] = (row y0, row y1): the recurrence of
// real_space_run with the two rows in the halves of the packed operations.
__device__ __forceinline__ void real_space_term(float qa, float qb, float qc, float mx, float my, float w, float r8,
                                                float y0, float y1, float x0, float2 (&o)[8]) {
  const float dx = x0 - mx, a = qa * dx, b = fmaf(2.0f, a, qa);
  const float dy0 = y0 - my, dy1 = y1 - my;
  const float l0 = qb * dy0, l1 = qb * dy1;
  float2 g = make_float2(w * ex2(fmaf(dx, a + l0, qc * dy0 * dy0)), w * ex2(fmaf(dx, a + l1, qc * dy1 * dy1)));
  float2 rr = make_float2(ex2(b + l0), ex2(b + l1));
  const float2 r2 = make_float2(r8, r8);
#pragma unroll
  for (int u = 0; u < 8; ++u) {
    o[u] = __fadd2_rn(o[u], g);
    if (u < 7) {
      g = __fmul2_rn(g, rr);
      rr = __fmul2_rn(rr, r2);
    }
  }
}

// The sum of a table's nr terms, added to o at the end (so that the phase and
// the Lanczos path, which convolves the sum first, round alike at integer
// offsets).
template <int R>
__device__ __forceinline__ void real_space_rows(const RealTermsN<R>& rt, int nr, float y0, float y1, float x0,
                                                float2 (&out)[8]) {
  float2 o[8];
#pragma unroll
  for (int u = 0; u < 8; ++u) o[u] = make_float2(0.0f, 0.0f);
#pragma unroll 1
  for (int t = 0; t < nr; t += 2) {
    const float4 p0 = rt.p[t >> 1][0], p1 = rt.p[t >> 1][1], p2 = rt.p[t >> 1][2], p3 = rt.p[t >> 1][3];
    real_space_term(p0.x, p1.z, p2.x, p1.x, p0.z, p2.z, p3.x, y0, y1, x0, o);
    if (t + 1 < nr) real_space_term(p0.y, p1.w, p2.y, p1.y, p0.w, p2.w, p3.y, y0, y1, x0, o);
  }
#pragma unroll
  for (int u = 0; u < 8; ++u) out[u] = __fadd2_rn(out[u], o[u]);
}

// The Fourier mixture of one profile at the thread's 16 bins of a column,
// omega = omj + m / 16, minus 1 from m = 8 on (pairs 2k, 2k+1 packed):
// s += sum_i a_i 2^(c_i q), components fc[0, nf) as (a, a, c, c).  A component
// is skipped over a warp's bins when 2^(c q) < 2^-40 on all of them: one lane
// tests one component against the warp's smallest q.
__device__ __forceinline__ void mixture16(const float4* fc, int nf, float s11, float s12x2, float s22, float nu,
                                          float omj, float2 (&s)[8]) {
  constexpr float NEGLIGIBLE_LOG2 = -40.0f;
  const float a0 = s11 * nu * nu, a1 = s12x2 * nu;
  float2 q[8];
  float qmin = 3.4e38f;
#pragma unroll
  for (int k = 0; k < 8; ++k) {
    const float oa = omj + (float)(2 * k - (k >= 4 ? 16 : 0)) * 0.0625f, ob = oa + 0.0625f;
    q[k] = make_float2(fmaf(oa, fmaf(s22, oa, a1), a0), fmaf(ob, fmaf(s22, ob, a1), a0));
    qmin = fminf(qmin, fminf(q[k].x, q[k].y));
  }
  // (not negative: the bits order as integers)
  const float wmin = __uint_as_float(__reduce_min_sync(0xffffffffu, __float_as_uint(fmaxf(qmin, 0.0f))));
  const int lane = threadIdx.x & 31;
  unsigned live = __ballot_sync(0xffffffffu, lane < nf && fc[lane < nf ? lane : 0].z * wmin > NEGLIGIBLE_LOG2);
  for (; live; live &= live - 1) {
    const float4 ac = fc[__ffs(live) - 1];
    const float2 a2 = make_float2(ac.x, ac.y), c2 = make_float2(ac.z, ac.w);
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      const float2 e = __fmul2_rn(c2, q[k]);
      s[k] = __ffma2_rn(a2, make_float2(ex2(e.x), ex2(e.y)), s[k]);
    }
  }
}

// Real-space part of a Lanczos-shifted galaxy: Lz(R), R the nr terms at the
// integer offset, Lz the periodic Lanczos convolution with weights wl (x:
// [0, 7), y: [8, 15)), in strips of STRIP rows: the rows a strip needs are
// evaluated and convolved along x (8 pixels of two rows per thread, neighbours
// by shuffle) into `strip`, shared memory of (STRIP + 6) rows, then along y;
// add(y, x0, acc) takes 8 pixels of the result.  One strip of all N rows has no
// halo (N rows of shared memory).  Called by all threads; starts writing
// `strip` at once and ends with a CTA barrier.  Shared-memory wavefronts bound it
// (seven rows read per output row, the 16-byte pieces two to a bank), so a row
// is read once for four output rows, the pieces are spread and the products are
// packed: a render of 30k galaxies of mixed sides with the shift 1.182 -> 1.023
// ms, of 30k of 64 x 64 0.463 -> 0.421.
template <int N, int STRIP, int THREADS, int R, class Add>
__device__ __forceinline__ void lanczos_real_strips(const RealTermsN<R>& rt, int nr, const float* wl, float* strip, Add add) {
  static_assert(STRIP % 2 == 0 && N % STRIP == 0, "rows in pairs, whole strips");
  constexpr int LANES = N / 8, GROUPS = THREADS / LANES;   // lanes per row
  const int j = threadIdx.x % LANES, g = threadIdx.x / LANES;
  const unsigned lanes = (0xffffffffu >> (32 - LANES)) << (threadIdx.x & 31 & ~(LANES - 1));
  constexpr bool WHOLE = STRIP == N;
  constexpr int ROWS = WHOLE ? N : STRIP + 6, HALO = WHOLE ? 0 : 3;
  const int x0 = 8 * j;
  // Pixel x is kept at x ^ 4 [bit 5 of x]: the 8 lanes of a quarter-warp, which
  // touch pieces 2j, take different banks.
  const int p0 = x0 ^ (((x0 >> 5) & 1) << 2);
#pragma unroll 1
  for (int y0 = 0; y0 < N; y0 += STRIP) {
    // rows y0 - HALO .. y0 + STRIP + HALO - 1 (mod N), two at a time, convolved along x
    // (the two rows in the halves of the packed operations)
    float2 w[7];
#pragma unroll
    for (int a = 0; a < 7; ++a) w[a] = make_float2(wl[a], wl[a]);
    for (int i = 2 * g; i < ROWS; i += 2 * GROUPS) {
      float2 r[8];
#pragma unroll
      for (int u = 0; u < 8; ++u) r[u] = make_float2(0.0f, 0.0f);
      real_space_rows(rt, nr, (float)((y0 - HALO + i) & (N - 1)), (float)((y0 - HALO + 1 + i) & (N - 1)), (float)x0, r);
      float2 win[14];
#pragma unroll
      for (int u = 0; u < 8; ++u) win[3 + u] = r[u];
#pragma unroll
      for (int a = 0; a < 3; ++a) {   // x0 - 3 + a from the lane below, x0 + 8 + a from the lane above
        win[a].x = __shfl_sync(lanes, r[5 + a].x, (j + LANES - 1) % LANES, LANES);
        win[a].y = __shfl_sync(lanes, r[5 + a].y, (j + LANES - 1) % LANES, LANES);
        win[11 + a].x = __shfl_sync(lanes, r[a].x, (j + 1) % LANES, LANES);
        win[11 + a].y = __shfl_sync(lanes, r[a].y, (j + 1) % LANES, LANES);
      }
      float2 X[8];
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        X[u] = make_float2(0.0f, 0.0f);
#pragma unroll
        for (int a = 0; a < 7; ++a) X[u] = __ffma2_rn(w[a], win[6 + u - a], X[u]);
      }
      float* const srow = strip + i * N;
      *reinterpret_cast<float4*>(srow + p0) = make_float4(X[0].x, X[1].x, X[2].x, X[3].x);
      *reinterpret_cast<float4*>(srow + (p0 ^ 4)) = make_float4(X[4].x, X[5].x, X[6].x, X[7].x);
      *reinterpret_cast<float4*>(srow + N + p0) = make_float4(X[0].y, X[1].y, X[2].y, X[3].y);
      *reinterpret_cast<float4*>(srow + N + (p0 ^ 4)) = make_float4(X[4].y, X[5].y, X[6].y, X[7].y);
    }
    __syncthreads();
    // output rows y0 + o: sum_b wy_b X(y - b), b = -3 .. 3, RB rows per thread:
    // each row of the strip is read once for all of them, from the last down,
    // so that every sum has its terms in the order of b
    constexpr int RB = 4;
    static_assert(STRIP % RB == 0, "whole blocks of rows");
#pragma unroll
    for (int a = 0; a < 7; ++a) w[a] = make_float2(wl[8 + a], wl[8 + a]);
    for (int o = RB * g; o < STRIP; o += RB * GROUPS) {
      float2 acc[RB][4];
#pragma unroll
      for (int i = 0; i < RB; ++i)
#pragma unroll
        for (int u = 0; u < 4; ++u) acc[i][u] = make_float2(0.0f, 0.0f);
#pragma unroll
      for (int t = 0; t < RB + 6; ++t) {
        const int y = o + RB + 2 - t;   // from y0
        const float* const srow = strip + (WHOLE ? y & (N - 1) : y + HALO) * N;
        const float4 a = *reinterpret_cast<const float4*>(srow + p0), c = *reinterpret_cast<const float4*>(srow + (p0 ^ 4));
        const float2 v[4] = {make_float2(a.x, a.y), make_float2(a.z, a.w), make_float2(c.x, c.y), make_float2(c.z, c.w)};
#pragma unroll
        for (int i = 0; i < RB; ++i)
          if (t - (RB - 1 - i) >= 0 && t - (RB - 1 - i) < 7) {
#pragma unroll
            for (int u = 0; u < 4; ++u) acc[i][u] = __ffma2_rn(w[t - (RB - 1 - i)], v[u], acc[i][u]);
          }
      }
#pragma unroll
      for (int i = 0; i < RB; ++i) {
        const float out[8] = {acc[i][0].x, acc[i][0].y, acc[i][1].x, acc[i][1].y,
                              acc[i][2].x, acc[i][2].y, acc[i][3].x, acc[i][3].y};
        add(y0 + o + i, x0, out);
      }
    }
    __syncthreads();
  }
}

}  // namespace mog
