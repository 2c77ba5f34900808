// Length-N transforms with 16 values per thread (N = 16 T, T threads of one
// warp each): a radix-16 pass in registers, one exchange through shared
// memory, then 16 / T radix-T transforms in registers.  Against the radix-8
// Stockham passes of common.cuh (8 values per thread) a 128- or 256-point
// transform has one exchange instead of two.
#pragma once

#include "common.cuh"

namespace mog {

// ------------------------------------------------------------------------
// 16-point DFT, sign S, as 4 x 4: input m = a + 4 d, output k = b + 4 c,
// w16^(m k) = w16^(a b) w4^(a c) w4^(d b).  Output k is left at v[at16(k)].
// ------------------------------------------------------------------------
__host__ __device__ constexpr int at16(int k) { return (k >> 2) + 4 * (k & 3); }

template <int S>
__device__ __forceinline__ void dft4_at(float2& v0, float2& v1, float2& v2, float2& v3) {
  const float2 a = padd(v0, v2), b = psub(v0, v2);
  const float2 c = padd(v1, v3), d = mul_si<S>(psub(v1, v3));
  v0 = padd(a, c);
  v2 = psub(a, c);
  v1 = cadd(b, d);
  v3 = csub(b, d);
}

template <int S>
__device__ __forceinline__ void dft16(float2* v) {
  constexpr float R = 0.70710678118654752440f, C1 = 0.92387953251128675613f, S1 = 0.38268343236508977173f;
#pragma unroll
  for (int a = 0; a < 4; ++a) dft4_at<S>(v[a], v[a + 4], v[a + 8], v[a + 12]);
  // v[a + 4 b] *= w16^(a b): exponents 1 2 3, 2 4 6, 3 6 9
  auto w1 = [&](float2 z, float c, float s) {   // z (c + S i s)
    return make_float2(fmaf(c, z.x, -S * s * z.y), fmaf(c, z.y, S * s * z.x));
  };
  v[5] = w1(v[5], C1, S1);
  v[9] = make_float2(R * (v[9].x - S * v[9].y), R * (v[9].y + S * v[9].x));
  v[13] = w1(v[13], S1, C1);
  v[6] = make_float2(R * (v[6].x - S * v[6].y), R * (v[6].y + S * v[6].x));
  v[10] = mul_si<S>(v[10]);
  v[14] = make_float2(R * (-v[14].x - S * v[14].y), R * (-v[14].y + S * v[14].x));
  v[7] = w1(v[7], S1, C1);
  v[11] = make_float2(R * (-v[11].x - S * v[11].y), R * (-v[11].y + S * v[11].x));
  v[15] = w1(v[15], -C1, -S1);
#pragma unroll
  for (int b = 0; b < 4; ++b) dft4_at<S>(v[4 * b], v[4 * b + 1], v[4 * b + 2], v[4 * b + 3]);
}

// ------------------------------------------------------------------------
// The transform.  Thread j of the group enters with x[j + T m] in v[m] and
// leaves with X[k1 + 16 k2], k1 = j + T q, in v[fft16_at<N>(q, k2)]
// (q < 16 / T, k2 < T).  Between the passes element (k1, j) of the first one's
// output goes from thread j to thread k1 mod T through shared memory, at
// write(k1) for thread j and read(q, i) for element (j + T q, i).
// ------------------------------------------------------------------------
template <int N>
__host__ __device__ constexpr int fft16_threads() { return N / 16; }
template <int N>
__host__ __device__ constexpr int fft16_at(int q, int k2) {
  constexpr int T = fft16_threads<N>();
  return T == 16 ? at16(k2) : q * T + k2;
}

// Twiddles of thread j: tw[k1 - 1] = w_N^(j k1), k1 = 1..15 (w_N = e^{2 pi i / N};
// forward transforms use the conjugate).  A thread's role is fixed for the
// whole kernel, so they stay in registers.
template <int N>
__device__ __forceinline__ void fft16_twiddles(int j, float2 (&tw)[15]) {
#pragma unroll
  for (int k1 = 1; k1 < 16; ++k1) sincospif(2.0f * (float)(j * k1) / (float)N, &tw[k1 - 1].y, &tw[k1 - 1].x);
}

// `written` runs when the exchange's writes, which depend on every input of
// the thread, have been issued.
struct Nothing {
  __device__ __forceinline__ void operator()() const {}
};
template <int N, int S, class Write, class Read, class Written = Nothing>
__device__ __forceinline__ void fft16(const float2 (&tw)[15], float2 (&v)[16], Write write, Read read,
                                      Written written = Written()) {
  constexpr int T = fft16_threads<N>();
  dft16<S>(v);
#pragma unroll
  for (int k1 = 0; k1 < 16; ++k1) {
    float2 x = v[at16(k1)];
    if (k1 > 0) x = (S > 0) ? cmul(x, tw[k1 - 1]) : cmulc(x, tw[k1 - 1]);
    *write(k1) = x;
  }
  written();
  __syncwarp();
#pragma unroll
  for (int q = 0; q < 16 / T; ++q)
#pragma unroll
    for (int i = 0; i < T; ++i) v[q * T + i] = *read(q, i);
  __syncwarp();   // the exchange's place may be written again
#pragma unroll
  for (int q = 0; q < 16 / T; ++q) {
    if constexpr (T == 16) dft16<S>(v);
    else if constexpr (T == 8) dft8<S>(v + q * T);
    else if constexpr (T == 4) dft4<S>(v + q * T);
    else dft2<S>(v[q * T], v[q * T + 1]);
  }
}

// 16-byte asynchronous copy global -> shared of the issuing thread (waited
// for with async_copy_wait by that thread, then published by a barrier).
__device__ __forceinline__ void async_copy16(void* dst_smem, const void* src_gmem) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_u32(dst_smem)), "l"(src_gmem) : "memory");
}
__device__ __forceinline__ void async_copy_wait() { asm volatile("cp.async.wait_all;" ::: "memory"); }

}  // namespace mog
