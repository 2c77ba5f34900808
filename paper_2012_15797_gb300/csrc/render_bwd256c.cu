// Adjoint of 256 x 256 patches for small batches (gradients w.r.t. flux, x, y,
// log r_e, e1, e2 and optionally the Sersic index; the contraction of
// render_bwd.cu, see its header): one galaxy at a time per cluster of four
// 256-thread CTAs, 16 values per thread (fft16.cuh).  A CTA of
// render_bwd256.cu takes about 100 us for a galaxy, whatever the batch; when
// there are fewer galaxies than CTAs fit, spreading one over four SMs is what
// shortens the call (one galaxy 88 -> 29 us, 40 139 -> 47, 100 143 -> 81).
//
//   real      analytic real-space derivatives over the CTA's share of the pixels
//   rows      forward FFTs of the CTA's 32 row pairs (p, p + N/2), packed as
//             g[p] + i g[p + N/2], their 256 outputs left in shared memory
//   columns   each thread gathers the two elements k and N - k of its 8 row pairs
//             from the CTAs that hold them (distributed shared memory), untangles
//             them into the two rows' spectra, forward FFT along y, contraction
//             with the mixture's derivatives
//   reduce    warp shuffles, the warps' sums sent to the leading CTA
// Two cluster barriers per galaxy: rows complete, sums complete.
#include "cluster.cuh"
#include "fft16.cuh"
#include "internal.h"

namespace mog {

namespace {

constexpr int N = 256;
constexpr int T = fft16_threads<N>();   // threads per transform
constexpr int CL = 4;                   // CTAs per galaxy
constexpr int KL = N / 2 / CL;          // row pairs (and columns) per CTA
constexpr int THREADS = 256;
constexpr int GROUPS = THREADS / T;
constexpr int ROUNDS = KL / GROUPS;
constexpr int WARPS = THREADS / 32;
constexpr int LS = psf_lstride(N);
constexpr int PSF_ELEMS = psf_spec_elems(N);
constexpr int B = bucket_of(N);
constexpr int EX = T + 1;               // exchange element (k1, i) at 17 k1 + i: conflict free both ways
constexpr int RS = 16 * EX;             // a group's work row
// Output k of the CTA's row pair pl at k SZ + pl: an odd stride for the 16 k
// that a half-warp writes; the 16 row pairs that it gathers lie side by side.
constexpr int SZ = KL + 1;

constexpr size_t off_z = 0;
constexpr size_t off_w = off_z + sizeof(float2) * N * SZ;
constexpr size_t off_py = off_w + sizeof(float2) * GROUPS * RS;
constexpr size_t off_nb = off_py + sizeof(float2) * N;   // rank 0: nu = 1/2 column, P phase
constexpr size_t off_ns = off_nb + sizeof(float2) * N;   // and the mixture sums
constexpr size_t off_rec = (off_ns + sizeof(float) * 4 * N + 15) & ~size_t(15);
// LZ: phase times slope response along omega; the nu = 1/2 column's P phase
// with the slopes along x and along y; the phases times response and slope
// response of the CTA's columns
constexpr size_t LZ_ELEMS = 3 * N + 2 * KL;
constexpr size_t off_terms = off_rec + 2 * sizeof(AdjRecord);
constexpr size_t off_red = off_terms + sizeof(AdjTerms);
constexpr size_t SMEM = off_red + sizeof(float) * 8 * CL * WARPS;
constexpr size_t off_lz = SMEM;
constexpr size_t SMEM_LZ = off_lz + sizeof(float2) * LZ_ELEMS;
static_assert(SMEM_LZ <= 227 * 1024, "shared memory of a CTA");

// WN: also d L / d(Sersic n), a seventh gradient per galaxy.  EIG: some PSF of
// the context is an eigen-PSF (its spectrum combined bin by bin where read).
// LZ: the gradient of the Lanczos variant's model (see render_bwd.cu).
template <bool WN, bool EIG, bool LZ>
__global__ void __launch_bounds__(THREADS, 1)
    render_bwd256c_kernel(RenderParams p, const float* __restrict__ grad_out, float* __restrict__ grad_params) {
  constexpr float INV_N = 1.0f / N;
  constexpr float TWO_PI = 2.0f * PI_F;
  constexpr int NACC = WN ? 7 : 6;
  extern __shared__ __align__(128) unsigned char smem[];
  float2* Z = reinterpret_cast<float2*>(smem + off_z);
  float2* W = reinterpret_cast<float2*>(smem + off_w);
  float2* py = reinterpret_cast<float2*>(smem + off_py);
  float2* nyb = reinterpret_cast<float2*>(smem + off_nb);
  float* nys = reinterpret_cast<float*>(smem + off_ns);
  AdjRecord* rec = reinterpret_cast<AdjRecord*>(smem + off_rec);
  AdjTerms& at = *reinterpret_cast<AdjTerms*>(smem + off_terms);
  float* red = reinterpret_cast<float*>(smem + off_red);   // rank 0: [CTA][warp][8]
  [[maybe_unused]] float2* pyd = reinterpret_cast<float2*>(smem + off_lz);
  [[maybe_unused]] float2* nybx = pyd + N;   // rank 0
  [[maybe_unused]] float2* nyby = pyd + 2 * N;
  [[maybe_unused]] float2* px = pyd + 3 * N;
  [[maybe_unused]] float2* pxd = px + KL;
  __shared__ float4 s_fa[KMAX], s_fc[KMAX], s_fd[KMAX];    // component tables of adj_mixture_sums
  __shared__ float s_lw[LZ ? ADJ_LW : 1];                  // Lanczos weights and slopes

  const int tid = threadIdx.x;
  const int f = tid / T, j = tid % T;
  const int rank = (int)cluster_rank();
  float2 tw[15];
  fft16_twiddles<N>(j, tw);
  float2* const w = W + f * RS;
  auto at_k1 = [&](int k1) { return w + k1 * EX + j; };
  auto at_i = [&](int, int i) { return w + j * EX + i; };
  const int count = p.bucket_count[B], first = p.bucket_start[B];
  auto sync_all = [&]() {
    cluster_arrive();
    cluster_wait();
  };
  sync_all();   // every CTA of the cluster runs: its shared memory may be accessed

  // Records have two buffers: the leading thread reads galaxy i's while others
  // load that of i + 1.  Everything else of i is last read before its second
  // cluster barrier.
  int buf = 0;
  for (int pos = blockIdx.x / CL; pos < count; pos += gridDim.x / CL, buf ^= 1) {
    if (tid < (int)(sizeof(AdjRecord) / 16))
      reinterpret_cast<float4*>(&rec[buf])[tid] =
          __ldg(reinterpret_cast<const float4*>(p.records + ((size_t)first + pos) * sizeof(AdjRecord)) + tid);
    __syncthreads();
    const AdjRecord& r = rec[buf];
    if (!r.ok) continue;   // uniform over the cluster: every CTA reads the same record
    const DevPsf& ps = p.psfs[r.psf];
    const float* pc = p.pcoef + ((size_t)first + pos) * PCOEF;
    const int k_eig = EIG ? ps.k_eig : 0;
    const float2* const psf_hat = ps.spec[B];
    const float* gpatch = grad_out + r.off;
    const int nrt = r.nrc * ps.k, nr2 = real_terms_padded(nrt);

    // ---- per-galaxy tables; the nu = 1/2 column for the CTA of column 0 ----
    [[maybe_unused]] const float* lwg = LZ ? p.lzw + ((size_t)first + pos) * ADJ_LW : nullptr;
    // a phase times the responses of the weights at `at` (and of their slopes, 8 on)
    auto shift = [&](float2 ph, int at, float fr, float2& slope) {
      float wv[7];
      load_weights(lwg, at + 8, wv);
      slope = cmul(ph, lanczos_slope_response(wv, fr));
      load_weights(lwg, at, wv);
      return cmul(ph, lanczos_response(wv, fr));
    };
    const int t1 = N, t2 = t1 + (rank == 0 ? N : 0), t3 = t2 + nr2, t4 = t3 + r.nf;
    for (int i = tid; i < t4 + (LZ ? KL : 0); i += THREADS) {
      if (i < t2) {
        const int l = i < t1 ? i : i - t1;
        const float om = (float)(l < N / 2 ? l : l - N) * INV_N;
        float2 phy;
        [[maybe_unused]] float2 phyd;
        sincospif(-2.0f * r.y * om, &phy.y, &phy.x);
        if constexpr (LZ) phy = shift(phy, 16, om, phyd);
        if (i < t1) {
          py[l] = phy;
          if constexpr (LZ) {
            pyd[l] = phyd;
            if (l < ADJ_LW) s_lw[l] = lwg[l];
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
        nyb[l] = cmul(pn, cmul(phx, phy));
        if constexpr (LZ) {
          nybx[l] = cmul(pn, cmul(phxd, phy));
          nyby[l] = cmul(pn, cmul(phx, phyd));
        }
        nys[4 * l + 0] = s;
        nys[4 * l + 1] = sq;
        nys[4 * l + 2] = sn;
        nys[4 * l + 3] = sd;
      } else if (i < t3) {
        const int t = i - t2;
        if (t < nrt) adj_real_term(r, ps.mog, ps.k, N, t, &at, k_eig > 0 ? pc + 8 : nullptr);
        else adj_real_term_zero(t, &at);
      } else if (!LZ || i < t4) {
        adj_component_tables(r, i - t3, s_fa, s_fc, s_fd);
      } else if constexpr (LZ) {
        const int kl = i - t4;
        const float nu = (rank * KL + kl) * INV_N;
        float2 ph;
        sincospif(-2.0f * r.x * nu, &ph.y, &ph.x);
        px[kl] = shift(ph, 0, nu, pxd[kl]);
      }
    }
    __syncthreads();

    float acc[7] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
    adj_real_space<N, WN, LZ>(gpatch, N, at, nr2, rank * THREADS + tid, CL * THREADS, acc, r.s11, r.s12, r.s22, s_lw);

    // ---- rows ----
    float2 v[16];
#pragma unroll 1
    for (int cc = 0; cc < ROUNDS; ++cc) {
      const int pl = cc * GROUPS + f;
      const float* ga = gpatch + (size_t)(rank * KL + pl) * N + j;
      const float* gb = ga + (N / 2) * N;
#pragma unroll
      for (int m = 0; m < 16; ++m) v[m] = make_float2(__ldg(ga + m * T), __ldg(gb + m * T));
      fft16<N, -1>(tw, v, at_k1, at_i);
      float2* const z = Z + j * SZ + pl;
#pragma unroll
      for (int k2 = 0; k2 < 16; ++k2) z[16 * k2 * SZ] = v[fft16_at<N>(0, k2)];
    }
    sync_all();   // every row pair's spectrum is there

    // ---- columns, contraction ----
#pragma unroll 1
    for (int cc = 0; cc < ROUNDS; ++cc) {
      const int k = rank * KL + cc * GROUPS + f;   // column nu = k / N (column 0: nu = 0 and 1/2 packed)
      // row pair p = j + 16 m lies in CTA m / 2; its rows p and p + N/2 have
      // spectra (Z[k] + conj Z[N-k]) / 2 and (Z[k] - conj Z[N-k]) / (2i)
      const uint32_t zk = smem_u32(Z + k * SZ + j), zn = smem_u32(Z + (k ? N - k : N / 2) * SZ + j);
#pragma unroll
      for (int m = 0; m < 8; ++m) {
        const float2 a = cluster_ld2(cluster_map(zk + 8 * 16 * (m & 1), m >> 1));
        const float2 b = cluster_ld2(cluster_map(zn + 8 * 16 * (m & 1), m >> 1));
        // rows' nu = 0 and nu = 1/2 values are real: packed as re + i im
        v[m] = k ? make_float2(0.5f * (a.x + b.x), 0.5f * (a.y - b.y)) : make_float2(a.x, b.x);
        v[m + 8] = k ? make_float2(0.5f * (a.y + b.y), -0.5f * (a.x - b.x)) : make_float2(a.y, b.y);
      }
      fft16<N, -1>(tw, v, at_k1, at_i);
      if (k == 0) {   // packed U[l], natural order
#pragma unroll
        for (int k2 = 0; k2 < 16; ++k2) w[j + 16 * k2] = v[fft16_at<N>(0, k2)];
      }
      __syncwarp();
      const float nu = k * INV_N, ck = k == 0 ? 1.0f : 2.0f;
      const float s11 = r.s11, s12x2 = 2.0f * r.s12, s22 = r.s22;
      const float a0 = s11 * nu * nu, a1 = s12x2 * nu;
      const int nf = r.nf;
      float2 pxk;
      [[maybe_unused]] const float2 pxdk = LZ ? pxd[cc * GROUPS + f] : make_float2(0.f, 0.f);
      if constexpr (LZ) pxk = px[cc * GROUPS + f];
      else sincospif(-2.0f * r.x * nu, &pxk.y, &pxk.x);
      constexpr int BH = 8;   // bins per sweep over the components
#pragma unroll
      for (int b0 = 0; b0 < 16; b0 += BH) {
        // l = j + 16 k2, omega = l / N, minus 1 from k2 = 8 on
        const float om0 = (float)j * INV_N - (b0 ? 0.5f : 0.0f);
        float2 qp[BH / 2], S[BH / 2], SQ[BH / 2], SN[BH / 2], SD[BH / 2];
#pragma unroll
        for (int i = 0; i < BH / 2; ++i) {
          const float oa = om0 + (float)(2 * i) * 0.0625f, ob = om0 + (float)(2 * i + 1) * 0.0625f;
          qp[i] = make_float2(fmaf(oa, fmaf(s22, oa, a1), a0), fmaf(ob, fmaf(s22, ob, a1), a0));
        }
        adj_mixture_sums<BH / 2, WN>(s_fa, s_fc, s_fd, nf, qp, S, SQ, SN, SD);
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
            z = contract_shift(pv, gk, ck, pxk, pxdk, py[l], pyd[l], s, acc);
            contract_shape(z.x, nu, om, s, sq, sn, acc);
          } else {
            z = cscale(cmulc(cmul(pv, cmul(pxk, py[l])), gk), ck);
            contract_bin(z, nu, om, s, sq, sn, acc);
          }
          if constexpr (WN) acc[6] = fmaf(z.x, sd, acc[6]);
          if (k == 0) {
            const float2 zh = cmulc(nyb[l], gn);
            if constexpr (LZ) {
              acc[1] = fmaf(fmaf(nybx[l].x, gn.x, nybx[l].y * gn.y), nys[4 * l], acc[1]);
              acc[2] = fmaf(fmaf(nyby[l].x, gn.x, nyby[l].y * gn.y), nys[4 * l], acc[2]);
              contract_shape(zh.x, 0.5f, om, nys[4 * l], nys[4 * l + 1], nys[4 * l + 2], acc);
            } else {
              contract_bin(zh, 0.5f, om, nys[4 * l], nys[4 * l + 1], nys[4 * l + 2], acc);
            }
            if constexpr (WN) acc[6] = fmaf(zh.x, nys[4 * l + 3], acc[6]);
          }
        }
      }
      __syncwarp();   // the group's reads of its work row are done
    }

    // ---- reduce and chain rule ----
    const uint32_t slot = cluster_map(smem_u32(red + (rank * WARPS + (tid >> 5)) * 8), 0);
#pragma unroll
    for (int c = 0; c < NACC; ++c) {
      float x = acc[c];
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
      if ((tid & 31) == 0) cluster_st(slot + 4 * c, x);
    }
    sync_all();   // the sums are there, and every gather of Z has returned
    if (rank == 0 && tid == 0) {
      float t[7] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
      for (int i = 0; i < CL * WARPS; ++i)
        for (int c = 0; c < NACC; ++c) t[c] += red[i * 8 + c];
      float* out = grad_params + r.gal * NACC;
      if constexpr (WN) out[6] = t[6];
      out[0] = t[0] / r.flux;
      out[1] = (LZ ? 1.0f : TWO_PI) * t[1];
      out[2] = (LZ ? 1.0f : TWO_PI) * t[2];
#pragma unroll
      for (int c = 0; c < 3; ++c) out[3 + c] = t[3] * r.dS[c][0] + t[4] * r.dS[c][1] + t[5] * r.dS[c][2];
    }
  }
}

}  // namespace

cudaError_t launch_render_bwd256_small(const RenderParams& p, const float* grad_out, float* grad_params, int num_sms,
                                       cudaStream_t s) {
  auto fn = p.lanczos ? (p.eigen ? (p.grad_n ? render_bwd256c_kernel<true, true, true> : render_bwd256c_kernel<false, true, true>)
                                 : (p.grad_n ? render_bwd256c_kernel<true, false, true> : render_bwd256c_kernel<false, false, true>))
                      : (p.eigen ? (p.grad_n ? render_bwd256c_kernel<true, true, false> : render_bwd256c_kernel<false, true, false>)
                                 : (p.grad_n ? render_bwd256c_kernel<true, false, false> : render_bwd256c_kernel<false, false, false>));
  const size_t smem = p.lanczos ? SMEM_LZ : SMEM;
  if (kernel_occupancy(reinterpret_cast<const void*>(fn), THREADS, smem) < 0) return cudaErrorInvalidConfiguration;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3((unsigned)(persistent_grid(p, 1, num_sms / CL) * CL));
  cfg.blockDim = dim3(THREADS);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = CL;
  at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, fn, p, grad_out, grad_params);
}

}  // namespace mog
