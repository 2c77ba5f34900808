// Gaussian-mixture fit of pixelized PSFs on the device: the mixture that the
// real-space half of the method convolves with (Section 2, Step 4 uses a
// Gaussian approximation of the PSF; Section 1 describes chi-squared fits of
// mixtures).  A cluster of CTAs per image runs Levenberg-Marquardt on
//   chi^2 = sum_p (sum_j w_j N(p - c - m_j; V_j) - image[p])^2,
// w_j = exp(lw_j), V_j = L L^T with L = [[exp(la), 0], [b, exp(lc)]], from a
// start set by the image's second moment.  Everything is FP32: J^T J and
// J^T r are summed over chunks of 256 pixels in pixel order and across chunks
// with compensated (Kahan) addition, chi^2 of a trial point over the pixels of
// equal index in their chunks likewise; the damped normal equations are solved
// by Cholesky after scaling by the diagonal, D^-1 (J^T J) D^-1 with unit
// diagonal (Marquardt's scaling), which keeps the factorisation well
// conditioned.  Every loop is bounded by the iteration count.
//
// A fit takes some hundred iterations, one after the other, so what counts is
// the time of one.  The chunks' sums do not depend on one another: the CTAs of
// a cluster take CPS chunks each at a time, keep their Jacobian rows in shared
// memory and form every chunk's products at once, a 4 x 4 tile of the matrix
// per thread and chunk; the leading CTA adds the chunks up in their order, so
// that the order of every sum is the same for any cluster size.  The Jacobian
// and its products are formed at accepted points only (at an unchanged one the
// sums stand).  One warp factorises and solves, a row of the matrix per lane in
// registers.  64 images of 64 x 64, k = 3: 49.6 -> 10.9 ms with the same bits
// (one CTA of 256 threads per image, its chunks one after the other, thread 0
// solving); what is left is the latency of an iteration, about 27 us.  With more
// images than SMs one large CTA per SM leaves it idle where a warp solves, which
// small images do not make up for: batches of them have CTAs of 256 threads, four
// per SM, with the same bits (3000 images of 24 x 24, k = 3: 131 ms with the first
// form, 144 on large CTAs, 60; k = 1: 1.29, 2.23, 1.12; 40 x 40, k = 3: 158, 138,
// 91; 1000 of 128 x 128 387, 267 on large CTAs, 297 on small ones).
#include <cooperative_groups.h>

#include "fft16.cuh"
#include "internal.h"

namespace mog {

namespace {

constexpr int CHUNK = 256;        // pixels
constexpr float TWO_PI_F = 6.283185307179586f;

// MANY: the form for batches of many small images.
template <int K, bool MANY>
struct FitCfg {
  static constexpr int P = 6 * K;             // parameters
  static constexpr int Q = (P + 1 + 3) & ~3;  // Jacobian row: parameters, the residual, padding
  static constexpr int NT = Q / 4;            // 4 x 4 tiles per side
  static constexpr int TILES = NT * (NT + 1) / 2;
  static constexpr int CPS = MANY ? 2 : K == 4 ? 4 : 8;  // chunks whose Jacobian rows a CTA holds
  // The pixels of several chunks are evaluated side by side (one after the
  // other by 256 threads, their latency was two thirds of an iteration).
  static constexpr int THREADS = MANY ? 256 : K == 4 ? 512 : 1024;
  static constexpr int MIN_CTAS = MANY ? 4 : 1;
  static constexpr int SIDE = THREADS / CHUNK;
  static_assert(TILES * CPS <= THREADS && TILES * 16 <= THREADS, "one tile per thread, one sum per thread");
};

template <int K, bool MANY>
struct FitShared {
  using C = FitCfg<K, MANY>;
  float J[C::CPS * CHUNK * C::Q];
  float res[C::CPS * CHUNK];           // residuals at the trial point
  float part[C::CPS][C::TILES * 16];   // products of each chunk, by tile
  float theta[C::P], trial[C::P];
  float sums[C::TILES * 16];           // the leading CTA's: J^T J, J^T r, chi^2, by tile
  float scale[C::P];                   // sqrt of the diagonal
  float red[CHUNK / 32];
  float lambda, chi;
  int done, accepted;
};

// Mixture value, and (with jac) the derivatives of one component's terms
// w.r.t. its six parameters, at offset (dx, dy) from the PSF centre.
__device__ __forceinline__ float eval_pixel(const float* th, int k, float dx, float dy, float* jac) {
  float model = 0.0f;
  for (int c = 0; c < k; ++c) {
    const float wgt = expf(th[6 * c]), mx = th[6 * c + 1], my = th[6 * c + 2];
    const float a = expf(th[6 * c + 3]), b = th[6 * c + 4], cc = expf(th[6 * c + 5]);
    const float vxx = a * a, vxy = a * b, vyy = b * b + cc * cc;
    const float det = vxx * vyy - vxy * vxy;   // = (a cc)^2 > 0
    const float idet = 1.0f / det;
    const float ex = dx - mx, ey = dy - my;
    const float ixx = vyy * idet, ixy = -vxy * idet, iyy = vxx * idet;
    const float ux = ixx * ex + ixy * ey, uy = ixy * ex + iyy * ey;
    const float g = expf(-0.5f * (ex * ux + ey * uy)) / (TWO_PI_F * a * cc);
    const float wg = wgt * g;
    model += wg;
    if (jac) {
      const float qxx = 0.5f * (ux * ux - ixx), qxy = 0.5f * (ux * uy - ixy), qyy = 0.5f * (uy * uy - iyy);
      jac[6 * c + 0] = wg;
      jac[6 * c + 1] = wg * ux;
      jac[6 * c + 2] = wg * uy;
      jac[6 * c + 3] = wg * (qxx * 2.0f * a * a + 2.0f * qxy * a * b);
      jac[6 * c + 4] = wg * (2.0f * qxy * a + qyy * 2.0f * b);
      jac[6 * c + 5] = wg * (qyy * 2.0f * cc * cc);
    }
  }
  return model;
}

// Sum over the first CHUNK threads (called by all).
__device__ float block_sum(float v, float* red) {
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  __syncthreads();
  if (lane == 0 && warp < CHUNK / 32) red[warp] = v;
  __syncthreads();
  float t = 0.0f;
  for (int i = 0; i < CHUNK / 32; ++i) t += red[i];
  return t;
}

// acc += x with the rounding error carried in comp (Kahan).
__device__ __forceinline__ void kahan_add(float& acc, float& comp, float x) {
  const float y = x - comp;
  const float t = acc + y;
  comp = (t - acc) - y;
  acc = t;
}

// Position in the tiled sums of the product of columns i <= j.
template <int K>
__device__ __forceinline__ int tiled(int i, int j) {
  const int ti = i >> 2, tj = j >> 2;
  return (ti * FitCfg<K, false>::NT - ti * (ti - 1) / 2 + tj - ti) * 16 + (i & 3) * 4 + (j & 3);
}

// The damped normal equations at S.theta (one warp of the leading CTA): with D
// = sqrt(diag J^T J), solve (D^-1 J^T J D^-1 + lambda I) z = -D^-1 J^T r by
// Cholesky; S.trial = theta + D^-1 z.  Lane i holds row i of the factor; every
// entry subtracts its products in ascending order.
template <int K, bool MANY>
__device__ __forceinline__ void solve_warp(FitShared<K, MANY>& S) {
  using C = FitCfg<K, MANY>;
  constexpr int P = C::P;
  constexpr unsigned ALL = 0xffffffffu;
  const int lane = threadIdx.x & 31;
  const int row = lane < P ? lane : P - 1;   // spare lanes repeat the last row
  const float Di = sqrtf(fmaxf(S.sums[tiled<K>(row, row)], 1e-30f));
  if (lane < P) S.scale[lane] = Di;
  __syncwarp();
  float L[P];
#pragma unroll
  for (int j = 0; j < P; ++j) {
    const int lo = min(row, j), hi = max(row, j);
    L[j] = row == j ? 1.0f + S.lambda : S.sums[tiled<K>(lo, hi)] / (S.scale[lo] * S.scale[hi]);
  }
  bool ok = true;
#pragma unroll
  for (int j = 0; j < P; ++j) {
    float v = L[j];
#pragma unroll
    for (int m = 0; m < j; ++m) v -= L[m] * __shfl_sync(ALL, L[m], j);
    const float d = __shfl_sync(ALL, v, j);
    ok = ok && d > 0.0f;
    const float r = sqrtf(d);
    L[j] = row == j ? r : v / r;
  }
  if (!ok) {   // uniform
    if (lane < P) S.trial[lane] = S.theta[lane];
    return;
  }
  float y = -S.sums[tiled<K>(row, P)] / Di;   // L y = -D^-1 J^T r
#pragma unroll
  for (int m = 0; m < P; ++m) {
    const float ym = __shfl_sync(ALL, y / L[m], m);
    y = row == m ? ym : row > m ? y - L[m] * ym : y;
  }
#pragma unroll
  for (int i = P - 1; i >= 0; --i) {   // L^T z = y
    float v = __shfl_sync(ALL, y, i);
#pragma unroll
    for (int m = i + 1; m < P; ++m) v -= __shfl_sync(ALL, L[i], m) * __shfl_sync(ALL, y, m);
    v = v / __shfl_sync(ALL, L[i], i);
    y = row == i ? v : y;
  }
  if (lane < P) S.trial[lane] = S.theta[lane] + y / Di;
}

template <int K, bool MANY>
__global__ void __launch_bounds__(FitCfg<K, MANY>::THREADS, FitCfg<K, MANY>::MIN_CTAS)
    psf_fit_kernel(const float* images, int h, int w, int k, int iters, float* rows_out, float* chi2_out) {
  using C = FitCfg<K, MANY>;
  constexpr int P = C::P, Q = C::Q;
  extern __shared__ __align__(16) unsigned char fit_smem[];
  FitShared<K, MANY>& S = *reinterpret_cast<FitShared<K, MANY>*>(fit_smem);
  const cooperative_groups::cluster_group cluster = cooperative_groups::this_cluster();
  const int rank = (int)cluster.block_rank(), ranks = (int)cluster.num_blocks();
  FitShared<K, MANY>& S0 = *cluster.map_shared_rank(&S, 0);   // the leading CTA's
  const bool lead = rank == 0;
  const int tid = threadIdx.x, px = tid % CHUNK, image = blockIdx.x / ranks;
  const float* img = images + (size_t)image * h * w;
  const int npix = h * w;
  const int cx = w / 2, cy = h / 2;
  const int chunks = (npix + CHUNK - 1) / CHUNK;
  const int steps = (chunks + ranks * C::CPS - 1) / (ranks * C::CPS);

  // start: weights and widths from the image sum and second moment
  if (lead) {
    float tot = 0.0f, mom = 0.0f;
    for (int p = tid; tid < CHUNK && p < npix; p += CHUNK) {
      const float dx = (float)(p % w - cx), dy = (float)(p / w - cy), v = img[p];
      tot += v;
      mom = fmaf(v, dx * dx + dy * dy, mom);
    }
    tot = block_sum(tot, S.red);
    mom = block_sum(mom, S.red);
    if (tid == 0) {
      const float scales[4] = {0.6f, 1.1f, 2.2f, 4.0f}, w0[4] = {0.55f, 0.35f, 0.08f, 0.015f};
      float wsum = 0.0f;
      for (int c = 0; c < K; ++c) wsum += w0[c];
      const float s = sqrtf(fmaxf(mom / (2.0f * tot), 0.25f));
      for (int c = 0; c < K; ++c) {
        S.theta[6 * c + 0] = logf(w0[c] / wsum * tot);
        S.theta[6 * c + 1] = 0.0f;
        S.theta[6 * c + 2] = 0.0f;
        S.theta[6 * c + 3] = logf(s * scales[c]);
        S.theta[6 * c + 4] = 0.0f;
        S.theta[6 * c + 5] = logf(s * scales[c]);
      }
      for (int i = 0; i < P; ++i) S.trial[i] = S.theta[i];
      S.lambda = 1e-3f;
      S.done = (tot > 0.0f && isfinite(tot)) ? 0 : 1;
      S.accepted = 1;
    }
  }
  cluster.sync();

  // residuals of this CTA's chunks of step s at the trial point
  auto residuals = [&](int s) {
    for (int lc = tid / CHUNK; lc < C::CPS; lc += C::SIDE) {
      const int p = ((s * ranks + rank) * C::CPS + lc) * CHUNK + px;
      if (p >= npix) break;
      const float dx = (float)(p % w - cx), dy = (float)(p / w - cy);
      S.res[lc * CHUNK + px] = eval_pixel(S.trial, k, dx, dy, nullptr) - img[p];
    }
  };
  // their Jacobian rows, with the residuals as column P
  auto jacobian = [&](int s) {
    for (int lc = tid / CHUNK; lc < C::CPS; lc += C::SIDE) {
      const int c = (s * ranks + rank) * C::CPS + lc, p = c * CHUNK + px;
      if (c >= chunks) break;
      float* row = S.J + (lc * CHUNK + px) * Q;
      if (p < npix) {
        const float dx = (float)(p % w - cx), dy = (float)(p / w - cy);
        const float model = eval_pixel(S.trial, k, dx, dy, row);
        row[P] = model - img[p];
      } else {
        for (int i = 0; i <= P; ++i) row[i] = 0.0f;
      }
      for (int i = P + 1; i < Q; ++i) row[i] = 0.0f;
    }
  };
  // products of this CTA's chunks of step s, summed over each chunk's pixels
  // in their order: one 4 x 4 tile of one chunk per thread
  auto products = [&](int s) {
    const int lc = tid / C::TILES, tile = tid % C::TILES;
    if (lc >= C::CPS || (s * ranks + rank) * C::CPS + lc >= chunks) return;
    int ti = 0, rem = tile;
    while (rem >= C::NT - ti) {   // bounded by NT
      rem -= C::NT - ti;
      ++ti;
    }
    const float4* const ri = reinterpret_cast<const float4*>(S.J + lc * CHUNK * Q) + ti;
    const float4* const rj = ri + rem;
    float acc[4][4] = {};
#pragma unroll 4
    for (int r = 0; r < CHUNK; ++r) {
      const float4 u = ri[r * (Q / 4)], v = rj[r * (Q / 4)];
      const float ui[4] = {u.x, u.y, u.z, u.w}, vj[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j] = fmaf(ui[i], vj[j], acc[i][j]);
    }
    float4* const d = reinterpret_cast<float4*>(&S.part[lc][tile * 16]);
#pragma unroll
    for (int i = 0; i < 4; ++i) d[i] = make_float4(acc[i][0], acc[i][1], acc[i][2], acc[i][3]);
  };

  // The trial point of the first pass is the start itself, accepted without a
  // test.  The conditions are the leading CTA's, read by every CTA between
  // two barriers.
  int it = 0;
  for (bool first = true;; first = false) {
    if (!lead && tid < P) S.trial[tid] = S0.trial[tid];
    __syncthreads();
    // ---- chi^2 at the trial point; accept, or raise the damping ----
    if (!first) {
      float c2 = 0.0f, cc2 = 0.0f;   // the leading CTA's
      for (int s = 0; s < steps; ++s) {
        residuals(s);
        cluster.sync();   // the residuals are there
        if (lead && tid < CHUNK)
          for (int rk = 0; rk < ranks; ++rk) {
            // a rank's chunks, loaded together, added in order
            const int c0 = (s * ranks + rk) * C::CPS;
            const float* const from = cluster.map_shared_rank(&S, rk)->res;
            float r[C::CPS];
#pragma unroll
            for (int i = 0; i < C::CPS; ++i) r[i] = (c0 + i) * CHUNK + tid < npix ? from[i * CHUNK + tid] : 0.0f;
#pragma unroll
            for (int i = 0; i < C::CPS; ++i)
              if ((c0 + i) * CHUNK + tid < npix) kahan_add(c2, cc2, r[i] * r[i]);
          }
        if (steps > 1) cluster.sync();   // they may be overwritten
      }
      if (lead) {
        c2 = block_sum(c2, S.red);
        if (tid == 0) {
          if (isfinite(c2) && c2 < S.chi) {
            const float rel = (S.chi - c2) / fmaxf(S.chi, 1e-30f);
            for (int i = 0; i < P; ++i) S.theta[i] = S.trial[i];
            S.lambda = fmaxf(S.lambda / 3.0f, 1e-7f);
            S.chi = c2;
            S.accepted = 1;
            if (rel < 1e-6f) S.done = 1;
          } else {
            S.accepted = 0;
            S.lambda *= 4.0f;
            if (S.lambda > 1e10f) S.done = 1;
          }
        }
      }
      ++it;
      cluster.sync();
    }
    const bool stop = S0.done || it >= iters, accepted = S0.accepted != 0;
    if (stop) break;   // uniform over the cluster
    // ---- J^T J, J^T r and chi^2 at an accepted point ----
    if (accepted) {
      float acc = 0.0f, comp = 0.0f;   // the leading CTA's, one sum per thread
      for (int s = 0; s < steps; ++s) {
        jacobian(s);
        __syncthreads();
        products(s);
        cluster.sync();
        if (lead && tid < C::TILES * 16)
          for (int rk = 0; rk < ranks; ++rk) {
            const int c0 = (s * ranks + rk) * C::CPS;
            const float* const from = cluster.map_shared_rank(&S, rk)->part[0];
            float x[C::CPS];
#pragma unroll
            for (int i = 0; i < C::CPS; ++i) x[i] = c0 + i < chunks ? from[i * C::TILES * 16 + tid] : 0.0f;
#pragma unroll
            for (int i = 0; i < C::CPS; ++i)
              if (c0 + i < chunks) kahan_add(acc, comp, x[i]);
          }
        if (steps > 1) cluster.sync();
      }
      if (lead) {
        if (tid < C::TILES * 16) S.sums[tid] = acc;
        __syncthreads();
        if (tid == 0) S.chi = S.sums[tiled<K>(P, P)];
      }
    }
    if (lead && tid < 32) {
      __syncwarp();
      solve_warp<K, MANY>(S);
    }
    cluster.sync();   // the trial point is there
  }

  // ---- output rows (w, mx, my, vxx, vxy, vyy), decreasing weight ----
  if (lead && tid == 0) {
    int order[K];
    for (int c = 0; c < K; ++c) order[c] = c;
    for (int a = 0; a < K; ++a)
      for (int b = a + 1; b < K; ++b)
        if (S.theta[6 * order[b]] > S.theta[6 * order[a]]) {
          const int t = order[a];
          order[a] = order[b];
          order[b] = t;
        }
    float* out = rows_out + (size_t)image * K * 6;
    for (int c = 0; c < K; ++c) {
      const float* t = S.theta + 6 * order[c];
      const float a = expf(t[3]), b = t[4], cc = expf(t[5]);
      out[6 * c + 0] = expf(t[0]);
      out[6 * c + 1] = t[1];
      out[6 * c + 2] = t[2];
      out[6 * c + 3] = a * a;
      out[6 * c + 4] = a * b;
      out[6 * c + 5] = b * b + cc * cc;
    }
    if (chi2_out) chi2_out[image] = S.chi;
  }
  cluster.sync();   // no CTA ends while another may read its shared memory
}

template <int K, bool MANY>
cudaError_t launch_fit_as(const float* images, int count, int h, int w, int iters, float* rows, float* chi2, int cl,
                          cudaStream_t s) {
  using C = FitCfg<K, MANY>;
  constexpr size_t SMEM = sizeof(FitShared<K, MANY>);
  if (kernel_occupancy(reinterpret_cast<const void*>(psf_fit_kernel<K, MANY>), C::THREADS, SMEM) < 0)
    return cudaErrorInvalidConfiguration;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3((unsigned)count * cl);
  cfg.blockDim = dim3(C::THREADS);
  cfg.dynamicSmemBytes = SMEM;
  cfg.stream = s;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = cl;
  at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, psf_fit_kernel<K, MANY>, images, h, w, K, iters, rows, chi2);
}

template <int K>
cudaError_t launch_fit(const float* images, int count, int h, int w, int iters, float* rows, float* chi2,
                       cudaStream_t s) {
  int device = 0, sms = 0;
  cudaError_t e = cudaGetDevice(&device);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, device);
  if (e != cudaSuccess) return e;
  const int64_t chunks = ((int64_t)h * w + CHUNK - 1) / CHUNK;
  // Many small images: CTAs of 256 threads, four per SM, so that one computes
  // while another waits or solves (see the header).  From three images per SM on
  // (608 of 24 x 24, k = 3: 12.3 ms against 31; 304 of 40 x 40 20.7 against 19.1);
  // larger images keep the large CTAs, whose iterations are shorter.  So do most
  // fits with two components, where some images take many more iterations than
  // the others and the call waits for them (3000 of 40 x 40: 24 ms against 20.5).
  if constexpr (K < 4) {
    if (count > (K == 2 ? 12 : 3) * sms && (chunks <= (K == 2 ? 5 : 24) || (K == 1 && count > 12 * sms)))
      return launch_fit_as<K, true>(images, count, h, w, iters, rows, chi2, 1, s);
  }
  // As many CTAs per image (1, 2, 4 or 8) as the SMs hold at once and the
  // image has chunks for.
  constexpr int CPS = FitCfg<K, false>::CPS;
  const int64_t steps = (chunks + CPS - 1) / CPS;
  int cl = 1;
  while (cl < 8 && (int64_t)count * cl * 2 <= sms && cl < steps) cl *= 2;
  return launch_fit_as<K, false>(images, count, h, w, iters, rows, chi2, cl, s);
}

}  // namespace

cudaError_t launch_psf_fit(const float* images, int count, int h, int w, int k, int iters, float* rows,
                           float* chi2, cudaStream_t s) {
  switch (k) {
    case 1: return launch_fit<1>(images, count, h, w, iters, rows, chi2, s);
    case 2: return launch_fit<2>(images, count, h, w, iters, rows, chi2, s);
    case 3: return launch_fit<3>(images, count, h, w, iters, rows, chi2, s);
    case 4: return launch_fit<4>(images, count, h, w, iters, rows, chi2, s);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace mog
