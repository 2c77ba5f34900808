// Adjoint of 256 x 256 patches: what the kernel of one CTA per galaxy
// (render_bwd256.cu) and the one of a cluster per galaxy (render_bwd256c.cu)
// share.  A galaxy's work is the same four parts in both, part i with the row
// pairs and columns 32 i .. 32 i + 31 and every fourth group of runs of pixels,
// 256 threads to a part: the cluster gives each part to a CTA, the other kernel
// takes them one after the other.  Every operation and the order of every sum
// is the same, so a galaxy's gradients do not depend on the kernel, and with it
// on how many other galaxies are in the call.
#pragma once

#include "fft16.cuh"
#include "internal.h"

namespace mog {
namespace bwd256 {

constexpr int N = 256;
constexpr int NP = N / 2;               // row pairs (p, p + N/2), columns
constexpr int T = fft16_threads<N>();   // 16 threads per transform
constexpr int PARTS = 4;
constexpr int KL = NP / PARTS;          // row pairs and columns of a part
constexpr int THREADS = 256;
constexpr int GROUPS = THREADS / T;
constexpr int ROUNDS = KL / GROUPS;     // transforms of one direction per thread group and part
constexpr int WARPS = THREADS / 32;
constexpr int LS = psf_lstride(N);
constexpr int PSF_ELEMS = psf_spec_elems(N);
constexpr int B = bucket_of(N);
constexpr int EX = T + 1;               // exchange element (k1, i) at 17 k1 + i: conflict free both ways
constexpr float INV_N = 1.0f / N;

// Per-galaxy tables in shared memory.  LZ: `px`, `py` times the Lanczos response
// of the weights, `pxd`, `pyd` times that of their slopes; nybx, nyby: the nu =
// 1/2 column with the slopes along x and along y.
struct Tables {
  float2 *py, *px;     // phase along omega [N] and nu [columns]
  float2* nyb;         // nu = 1/2 column: P phase
  float* nys;          // and the mixture sums, [l][4]: S, Sq, Sn, Sd
  float2 *pyd, *pxd, *nybx, *nyby;
  AdjTerms* at;
  float4 *fa, *fc, *fd;   // component tables of adj_mixture_sums
  float* lw;              // Lanczos weights and slopes
};

// Writes them (thread tid of `threads`): phases of columns k0 .. k0 + cols - 1,
// the nu = 1/2 column if `half`.
template <bool WN, bool EIG, bool LZ>
__device__ __forceinline__ void make_tables(const Tables& t, const AdjRecord& r, const DevPsf& ps, const float* pc,
                                            const float* lwg, int k0, int cols, bool half, int tid,
                                            int threads) {
  const int k_eig = EIG ? ps.k_eig : 0;
  const float2* const psf_hat = ps.spec[B];
  const int nrt = r.nrc * ps.k, nr2 = real_terms_padded(nrt);
  // a phase times the responses of the weights at `at` (and of their slopes, 8 on)
  auto shift = [&](float2 ph, int at, float fr, float2& slope) {
    float wv[7];
    load_weights(lwg, at + 8, wv);
    slope = cmul(ph, lanczos_slope_response(wv, fr));
    load_weights(lwg, at, wv);
    return cmul(ph, lanczos_response(wv, fr));
  };
  const int t1 = N, t2 = t1 + (half ? N : 0), t3 = t2 + cols, t4 = t3 + nr2;
  for (int i = tid; i < t4 + r.nf; i += threads) {
    if (i < t2) {
      const int l = i < t1 ? i : i - t1;
      const float om = (float)(l < N / 2 ? l : l - N) * INV_N;
      float2 phy;
      [[maybe_unused]] float2 phyd;
      sincospif(-2.0f * r.y * om, &phy.y, &phy.x);
      if constexpr (LZ) phy = shift(phy, 16, om, phyd);
      if (i < t1) {
        t.py[l] = phy;
        if constexpr (LZ) {
          t.pyd[l] = phyd;
          if (l < ADJ_LW) t.lw[l] = lwg[l];
        }
        continue;
      }
      const float q = fmaf(om, fmaf(r.s22, om, r.s12), 0.25f * r.s11);
      float s = 0.0f, sq = 0.0f, sn = 0.0f, sd = 0.0f;
      for (int c = 0; c < r.nf; ++c) {
        const float e = ex2(r.fcoef[c] * q);
        s = fmaf(r.famp[c], e, s);
        sq = fmaf(r.fq[c], e, sq);
        sn = fmaf(r.fn[c], e, sn);
        if constexpr (WN) sd = fmaf(fmaf(r.fdq[c], q, r.fdn[c]), e, sd);
      }
      float2 phx;
      [[maybe_unused]] float2 phxd;
      sincospif(-r.x, &phx.y, &phx.x);
      if constexpr (LZ) phx = shift(phx, 0, 0.5f, phxd);
      const int e = (N / 2) * LS + l;
      const float2 pn = k_eig > 0 ? eigen_bin(psf_hat, PSF_ELEMS, k_eig, pc, e) : __ldg(psf_hat + e);
      t.nyb[l] = cmul(pn, cmul(phx, phy));
      if constexpr (LZ) {
        t.nybx[l] = cmul(pn, cmul(phxd, phy));
        t.nyby[l] = cmul(pn, cmul(phx, phyd));
      }
      t.nys[4 * l + 0] = s;
      t.nys[4 * l + 1] = sq;
      t.nys[4 * l + 2] = sn;
      t.nys[4 * l + 3] = sd;
    } else if (i < t3) {
      const float nu = (float)(k0 + i - t2) * INV_N;
      float2 ph;
      sincospif(-2.0f * r.x * nu, &ph.y, &ph.x);
      if constexpr (LZ) ph = shift(ph, 0, nu, t.pxd[i - t2]);
      t.px[i - t2] = ph;
    } else if (i < t4) {
      const int u = i - t3;
      if (u < nrt) adj_real_term(r, ps.mog, ps.k, N, u, t.at, k_eig > 0 ? pc + 8 : nullptr);
      else adj_real_term_zero(u, t.at);
    } else {
      adj_component_tables(r, i - t4, t.fa, t.fc, t.fd);
    }
  }
}

// The elements a = Z[k], b = Z[N - k] (Z[N/2] for k = 0) of a row pair's packed
// transform as the values of column k in its rows p (lo) and p + N/2 (hi): their
// spectra are (Z[k] + conj Z[N-k]) / 2 and (Z[k] - conj Z[N-k]) / (2i); at k = 0
// the rows' nu = 0 and nu = 1/2 values are real, packed as re + i im.
__device__ __forceinline__ void untangle(int k, float2 a, float2 b, float2& lo, float2& hi) {
  lo = k ? make_float2(0.5f * (a.x + b.x), 0.5f * (a.y - b.y)) : make_float2(a.x, b.x);
  hi = k ? make_float2(0.5f * (a.y + b.y), -0.5f * (a.x - b.x)) : make_float2(a.y, b.y);
}

// Column nu = k / N (0: nu = 0 and 1/2 packed), rows j + 16 m in v[m]: forward
// transform along y, contraction with the mixture's derivatives.  w: the group's
// work row of 16 EX.  BH: bins per sweep over the components.
template <int BH, bool WN, bool EIG, bool LZ>
__device__ __forceinline__ void column(const Tables& t, const AdjRecord& r, const float2* psf_hat, int k_eig,
                                       const float* pc, int k, float2 pxk, float2 pxdk, const float2 (&tw)[15],
                                       float2 (&v)[16], float2* w, int j, float* acc) {
  fft16<N, -1>(
      tw, v, [&](int k1) { return w + k1 * EX + j; }, [&](int, int i) { return w + j * EX + i; });
  if (k == 0) {   // packed U[l], natural order
#pragma unroll
    for (int k2 = 0; k2 < 16; ++k2) w[j + 16 * k2] = v[fft16_at<N>(0, k2)];
  }
  __syncwarp();
  const float nu = k * INV_N, ck = k == 0 ? 1.0f : 2.0f;
  const float s11 = r.s11, s12x2 = 2.0f * r.s12, s22 = r.s22;
  const float a0 = s11 * nu * nu, a1 = s12x2 * nu;
  const int nf = r.nf;
#pragma unroll
  for (int b0 = 0; b0 < 16; b0 += BH) {
    // l = j + 16 k2, omega = l / N, minus 1 from k2 = 8 on
    const float om0 = (float)j * INV_N + (float)(b0 - (b0 >= 8 ? 16 : 0)) * 0.0625f;
    float2 qp[BH / 2], S[BH / 2], SQ[BH / 2], SN[BH / 2], SD[BH / 2];
#pragma unroll
    for (int i = 0; i < BH / 2; ++i) {
      const float oa = om0 + (float)(2 * i) * 0.0625f, ob = om0 + (float)(2 * i + 1) * 0.0625f;
      qp[i] = make_float2(fmaf(oa, fmaf(s22, oa, a1), a0), fmaf(ob, fmaf(s22, ob, a1), a0));
    }
    adj_mixture_sums<BH / 2, WN>(t.fa, t.fc, t.fd, nf, qp, S, SQ, SN, SD);
    [[maybe_unused]] float2 pe[BH];
    if constexpr (EIG)
      if (k_eig > 0)
        eigen_bins(psf_hat + k * LS + j, PSF_ELEMS, k_eig, pc, [&](int bb) { return 16 * (b0 + bb); }, pe);
#pragma unroll
    for (int bb = 0; bb < BH; ++bb) {
      const int k2 = b0 + bb, l = j + 16 * k2;
      const float om = om0 + (float)bb * 0.0625f;
      float2 gk = v[fft16_at<N>(0, k2)];
      float2 gn = make_float2(0.f, 0.f);
      if (k == 0) {
        const float2 u = w[l], un = w[(N - l) & (N - 1)];
        gk = make_float2(0.5f * (u.x + un.x), 0.5f * (u.y - un.y));
        gn = make_float2(0.5f * (u.y + un.y), -0.5f * (u.x - un.x));
      }
      const float s = (bb & 1) ? S[bb >> 1].y : S[bb >> 1].x;
      const float sq = (bb & 1) ? SQ[bb >> 1].y : SQ[bb >> 1].x;
      const float sn = (bb & 1) ? SN[bb >> 1].y : SN[bb >> 1].x;
      const float sd = (bb & 1) ? SD[bb >> 1].y : SD[bb >> 1].x;
      const float2 pv = (EIG && k_eig > 0) ? pe[bb] : __ldg(&psf_hat[k * LS + l]);
      float2 z;   // c_k conj(G) P phase
      if constexpr (LZ) {
        z = contract_shift(pv, gk, ck, pxk, pxdk, t.py[l], t.pyd[l], s, acc);
        contract_shape(z.x, nu, om, s, sq, sn, acc);
      } else {
        z = cscale(cmulc(cmul(pv, cmul(pxk, t.py[l])), gk), ck);
        contract_bin(z, nu, om, s, sq, sn, acc);
      }
      if constexpr (WN) acc[6] = fmaf(z.x, sd, acc[6]);
      if (k == 0) {
        const float2 zh = cmulc(t.nyb[l], gn);
        const float* const ny = t.nys + 4 * l;
        if constexpr (LZ) {
          acc[1] = fmaf(fmaf(t.nybx[l].x, gn.x, t.nybx[l].y * gn.y), ny[0], acc[1]);
          acc[2] = fmaf(fmaf(t.nyby[l].x, gn.x, t.nyby[l].y * gn.y), ny[0], acc[2]);
          contract_shape(zh.x, 0.5f, om, ny[0], ny[1], ny[2], acc);
        } else {
          contract_bin(zh, 0.5f, om, ny[0], ny[1], ny[2], acc);
        }
        if constexpr (WN) acc[6] = fmaf(zh.x, ny[3], acc[6]);
      }
    }
  }
  __syncwarp();   // the group's reads of its work row are done
}

// A warp's sum of acc[c], in every lane.
__device__ __forceinline__ float warp_sum(float x) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
  return x;
}

// One thread: the parts' and warps' sums red[part][warp][8] added up, the chain
// rule, the galaxy's gradients.
template <bool WN, bool LZ>
__device__ __forceinline__ void write_gradients(const AdjRecord& r, const float* red, float* grad_params) {
  constexpr int NACC = WN ? 7 : 6;
  constexpr float TWO_PI = 2.0f * PI_F;
  float t[7] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
  for (int i = 0; i < PARTS * WARPS; ++i)
    for (int c = 0; c < NACC; ++c) t[c] += red[i * 8 + c];
  float* out = grad_params + r.gal * NACC;
  if constexpr (WN) out[6] = t[6];
  out[0] = t[0] / r.flux;
  out[1] = (LZ ? 1.0f : TWO_PI) * t[1];
  out[2] = (LZ ? 1.0f : TWO_PI) * t[2];
#pragma unroll
  for (int c = 0; c < 3; ++c) out[3 + c] = t[3] * r.dS[c][0] + t[4] * r.dS[c][1] + t[5] * r.dS[c][2];
}

}  // namespace bwd256
}  // namespace mog
