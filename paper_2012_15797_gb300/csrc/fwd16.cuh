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
// add(y, x0, acc) takes 8 pixels of the result.  Called by all threads; starts
// writing `strip` at once and ends with a CTA barrier.
template <int N, int STRIP, int THREADS, int R, class Add>
__device__ __forceinline__ void lanczos_real_strips(const RealTermsN<R>& rt, int nr, const float* wl, float* strip, Add add) {
  static_assert(STRIP % 2 == 0 && N % STRIP == 0, "rows in pairs, whole strips");
  constexpr int LANES = N / 8, GROUPS = THREADS / LANES;   // lanes per row
  const int j = threadIdx.x % LANES, g = threadIdx.x / LANES;
  const unsigned lanes = (0xffffffffu >> (32 - LANES)) << (threadIdx.x & 31 & ~(LANES - 1));
  const int x0 = 8 * j;
  float wx[7], wy[7];
#pragma unroll
  for (int a = 0; a < 7; ++a) {
    wx[a] = wl[a];
    wy[a] = wl[8 + a];
  }
#pragma unroll 1
  for (int y0 = 0; y0 < N; y0 += STRIP) {
    // rows y0 - 3 .. y0 + STRIP + 2 (mod N), two at a time, convolved along x
    for (int i = 2 * g; i < STRIP + 6; i += 2 * GROUPS) {
      float2 r[8];
#pragma unroll
      for (int u = 0; u < 8; ++u) r[u] = make_float2(0.0f, 0.0f);
      real_space_rows(rt, nr, (float)((y0 - 3 + i) & (N - 1)), (float)((y0 - 2 + i) & (N - 1)), (float)x0, r);
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        float win[14];
#pragma unroll
        for (int u = 0; u < 8; ++u) win[3 + u] = h ? r[u].y : r[u].x;
#pragma unroll
        for (int a = 0; a < 3; ++a) {   // x0 - 3 + a from the lane below, x0 + 8 + a from the lane above
          win[a] = __shfl_sync(lanes, h ? r[5 + a].y : r[5 + a].x, (j + LANES - 1) % LANES, LANES);
          win[11 + a] = __shfl_sync(lanes, h ? r[a].y : r[a].x, (j + 1) % LANES, LANES);
        }
        float X[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) {
          float acc = 0.0f;
#pragma unroll
          for (int a = 0; a < 7; ++a) acc = fmaf(wx[a], win[3 + u - (a - 3)], acc);
          X[u] = acc;
        }
        float4* srow = reinterpret_cast<float4*>(strip + (i + h) * N + x0);
        srow[0] = make_float4(X[0], X[1], X[2], X[3]);
        srow[1] = make_float4(X[4], X[5], X[6], X[7]);
      }
    }
    __syncthreads();
    // output rows y0 + o: sum_b wy_b X(y - b), strip rows o + 3 - b
    for (int o = g; o < STRIP; o += GROUPS) {
      float acc[8];
#pragma unroll
      for (int u = 0; u < 8; ++u) acc[u] = 0.0f;
#pragma unroll
      for (int b = 0; b < 7; ++b) {
        const float4* srow = reinterpret_cast<const float4*>(strip + (o + 6 - b) * N + x0);
        const float4 p0 = srow[0], p1 = srow[1];
        const float v[8] = {p0.x, p0.y, p0.z, p0.w, p1.x, p1.y, p1.z, p1.w};
#pragma unroll
        for (int u = 0; u < 8; ++u) acc[u] = fmaf(wy[b], v[u], acc[u]);
      }
      add(y0 + o, x0, acc);
    }
    __syncthreads();
  }
}

}  // namespace mog
