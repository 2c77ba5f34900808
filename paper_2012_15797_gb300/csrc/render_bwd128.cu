// Fused adjoint of 128 x 128 patches with 16 values per thread (fft16.cuh):
// gradients of L w.r.t. (flux, x, y, log r_e, e1, e2) and optionally the Sersic
// index, given g = dL/d pixel (the sums are those of render_bwd.cu, see its
// header).  Two 256-thread CTAs per SM, one galaxy at a time per CTA, 8 threads
// per transform.
//
// The one large buffer is the N/2 rows of Z, in which everything is done in
// place:
//
//   staging   the patch, rows p and p + N/2 side by side in row p (bulk copies)
//   real      real-space derivatives; a group takes the runs of its own row pairs
//   rows      forward FFT of row pair p, packed as g[p] + i g[p + N/2], in row p
//   columns   a group gathers elements k and N - k of every row, untangles them
//             into the rows' spectra, forward FFT along y, exchanged in the places
//             it gathered from; contraction with the mixture's derivatives on
//             the 16 bins the thread ends with
//   reduce    warp shuffles, one thread applies the chain rule
//
// Three CTA barriers per galaxy: tables and patch there, rows done, sums there.
// Bound by latency and issue slots at the 16 warps per SM that 128 registers a
// thread leave.  Against 8 values per thread (two exchanges per transform, the
// spectra untangled through a second buffer, the patch read twice from L2): the
// 32.8k 128 x 128 galaxies of the 200k mixed workload 3.00 -> 2.76 ms, with the
// Sersic index 3.47 -> 3.17, Lanczos 5.46 -> 4.78.
#include "fft16.cuh"
#include "internal.h"

namespace mog {

namespace {

constexpr int N = 128;
constexpr int T = fft16_threads<N>();   // 8 threads per transform
constexpr int NP = N / 2;               // columns, row pairs
constexpr int ROUNDS = 2;               // transforms of one direction per thread group
constexpr int GROUPS = NP / ROUNDS;
constexpr int THREADS = GROUPS * T;     // 256
constexpr int WARPS = THREADS / 32;
constexpr int CTAS_PER_SM = 2;
constexpr int LS = psf_lstride(N);
constexpr int PSF_ELEMS = psf_spec_elems(N);
constexpr int B = bucket_of(N);
constexpr int RS = N + 16 / T;          // row stride of Z (float2), as in render_fwd128.cu

template <bool WN, bool LZ>
struct BCfg {
  static constexpr int NYS = WN ? 4 : 3;         // nu = 1/2 column sums per bin: S, Sq, Sn (and Sd)
  static constexpr size_t off_z = 0;
  static constexpr size_t off_py = off_z + sizeof(float2) * NP * RS;
  static constexpr size_t off_px = off_py + sizeof(float2) * N;
  static constexpr size_t off_nb = off_px + sizeof(float2) * NP;     // nu = 1/2 column: P phase
  static constexpr size_t off_ns = off_nb + sizeof(float2) * N;      // and the mixture sums
  // LZ: phase times slope response along omega and nu, and the nu = 1/2 column's
  // P phase with the slopes along x and along y
  static constexpr size_t off_lz = (off_ns + sizeof(float) * NYS * N + 15) & ~size_t(15);
  static constexpr size_t off_rec = off_lz + (LZ ? sizeof(float2) * (3 * N + NP) : 0);
  static constexpr size_t off_terms = off_rec + 3 * sizeof(AdjRecord);
  static constexpr size_t off_red = off_terms + sizeof(AdjTerms);
  static constexpr size_t off_bar = off_red + sizeof(float) * 8 * WARPS;
  static constexpr size_t SMEM = off_bar + sizeof(uint64_t);
  static_assert(CTAS_PER_SM * (SMEM + 1024 + 1024) <= 228 * 1024, "two CTAs share an SM's shared memory");
};

// Row pair of group f, as in render_fwd128.cu.
__device__ __forceinline__ int pair_of(int f) { return (f & ~7) | ((f & 1) << 2) | (f & 2) | ((f >> 2) & 1); }

// WN: also d L / d(Sersic n).  EIG: some PSF of the context is an eigen-PSF (its
// spectrum combined bin by bin where read).  LZ: the gradient of the Lanczos
// variant's model (see render_bwd.cu).
template <bool WN, bool EIG, bool LZ>
__global__ void __launch_bounds__(THREADS, CTAS_PER_SM)
    render_bwd128_kernel(RenderParams p, const float* __restrict__ grad_out, float* __restrict__ grad_params) {
  using C = BCfg<WN, LZ>;
  constexpr int NACC = WN ? 7 : 6;
  constexpr float INV_N = 1.0f / N;
  constexpr float TWO_PI = 2.0f * PI_F;
  extern __shared__ __align__(128) unsigned char smem[];
  float2* Z = reinterpret_cast<float2*>(smem + C::off_z);
  float2* py = reinterpret_cast<float2*>(smem + C::off_py);
  float2* px = reinterpret_cast<float2*>(smem + C::off_px);
  float2* nyb = reinterpret_cast<float2*>(smem + C::off_nb);
  float* nys = reinterpret_cast<float*>(smem + C::off_ns);
  [[maybe_unused]] float2* pyd = reinterpret_cast<float2*>(smem + C::off_lz);
  [[maybe_unused]] float2* nybx = pyd + N;
  [[maybe_unused]] float2* nyby = pyd + 2 * N;
  [[maybe_unused]] float2* pxd = pyd + 3 * N;
  AdjRecord* rec = reinterpret_cast<AdjRecord*>(smem + C::off_rec);   // [3]
  AdjTerms& at = *reinterpret_cast<AdjTerms*>(smem + C::off_terms);
  float* red = reinterpret_cast<float*>(smem + C::off_red);
  uint64_t* bar = reinterpret_cast<uint64_t*>(smem + C::off_bar);     // the patch
  __shared__ int s_first[2], s_pos;
  __shared__ float4 s_fa[KMAX], s_fc[KMAX], s_fd[KMAX];   // component tables of adj_mixture_sums
  __shared__ float s_lw[LZ ? ADJ_LW : 1];                 // Lanczos weights and slopes

  const int tid = threadIdx.x;
  const int f = tid / T, j = tid % T;
  float2 tw[15];
  fft16_twiddles<N>(j, tw);
  const int count = p.bucket_count[B], first = p.bucket_start[B];
  const unsigned char* records = p.records + (size_t)first * sizeof(AdjRecord);
  // the work queue, taken by thread 0; a position is published two galaxies ahead
  int q_next = 0, q_end = 0, q_ahead = 0;
  auto next_position = [&]() -> int {
    if (q_next >= q_end) {
      const int b0 = q_ahead;
      if (b0 >= count) return -1;
      q_next = b0;
      q_end = min(b0 + p.chunk, count);
      q_ahead = atomicAdd(&p.queue[B], p.chunk);
    }
    return q_next++;
  };
  auto load_record = [&](int b, int pos) {
    if (tid < (int)(sizeof(AdjRecord) / 16))
      async_copy16(reinterpret_cast<float4*>(&rec[b]) + tid,
                   reinterpret_cast<const float4*>(records + (size_t)pos * sizeof(AdjRecord)) + tid);
  };
  if (tid == 0) {
    mbar_init(bar, 1);
    q_ahead = atomicAdd(&p.queue[B], p.chunk);
    s_first[0] = next_position();
    s_first[1] = next_position();
  }
  __syncthreads();
  int pos = s_first[0], pos1 = s_first[1];
  if (pos >= 0) load_record(0, pos);
  async_copy_wait();
  __syncthreads();

  // Who waits for whom: the tables, the patch and Z of galaxy i are written
  // after every thread has passed the last barrier of i - 1, which follows all
  // reads of them; only thread 0 still reads (the sums, and the record of i - 1,
  // whose buffer is not written before the record of i + 2).
  uint32_t parity = 0;
  int b3 = 0;
  for (; pos >= 0;) {
    const AdjRecord& r = rec[b3];
    const int b3n = b3 == 2 ? 0 : b3 + 1;
    if (pos1 >= 0) load_record(b3n, pos1);
    int pos2 = -1;
    if (tid == 0) pos2 = next_position();
    const bool work = r.ok != 0;   // uniform
    const DevPsf& ps = p.psfs[work ? r.psf : 0];
    const float* pc = p.pcoef + ((size_t)first + pos) * PCOEF;
    const int k_eig = EIG ? ps.k_eig : 0;
    const float2* const psf_hat = ps.spec[B];
    const int nrt = work ? r.nrc * ps.k : 0, nr2 = real_terms_padded(nrt);
    bool landed = true;
    if (work) {
      // the patch: rows y and y + N/2 into the halves of row y of Z
      if (tid < 32) {
        if (tid == 0) mbar_expect_tx(bar, sizeof(float) * N * N);
        __syncwarp();
        for (int y = tid; y < N; y += 32)
          bulk_copy(reinterpret_cast<float*>(Z + (y & (NP - 1)) * RS) + (y >= NP ? N : 0),
                    grad_out + r.off + (size_t)y * N, sizeof(float) * N, bar);
      }
      // ---- per-galaxy tables ----
      [[maybe_unused]] const float* lwg = LZ ? p.lzw + ((size_t)first + pos) * ADJ_LW : nullptr;
      const float gx = r.x, gy = r.y;
      constexpr int t1 = N, t2 = 2 * N, t3 = t2 + NP;
      for (int i = tid; i < t3 + nr2 + r.nf; i += THREADS) {
        if (i < t2) {
          // phase along omega; the nu = 1/2 column: P phase and the mixture sums
          const int l = i < t1 ? i : i - t1;
          const float om = (float)(l < N / 2 ? l : l - N) * INV_N;
          float2 phy, phyd;
          sincospif(-2.0f * gy * om, &phy.y, &phy.x);
          if constexpr (LZ) {
            float w[7];
            load_weights(lwg, 24, w);
            phyd = cmul(phy, lanczos_slope_response(w, om));
            load_weights(lwg, 16, w);
            phy = cmul(phy, lanczos_response(w, om));
          }
          if (i < t1) {
            py[l] = phy;
            if constexpr (LZ) {
              pyd[l] = phyd;
              if (l < ADJ_LW) s_lw[l] = lwg[l];
            }
          } else {
            const float q = fmaf(om, fmaf(r.s22, om, r.s12), 0.25f * r.s11);
            float s = 0.0f, sq = 0.0f, sn = 0.0f, sd = 0.0f;
            for (int c = 0; c < r.nf; ++c) {
              const float e = ex2(r.fcoef[c] * q);
              s = fmaf(r.famp[c], e, s);
              sq = fmaf(r.fq[c], e, sq);
              sn = fmaf(r.fn[c], e, sn);
              if constexpr (WN) sd = fmaf(fmaf(r.fdq[c], q, r.fdn[c]), e, sd);
            }
            float2 phx, phxd;
            sincospif(-gx, &phx.y, &phx.x);
            if constexpr (LZ) {
              float w[7];
              load_weights(lwg, 8, w);
              phxd = cmul(phx, lanczos_slope_response(w, 0.5f));
              load_weights(lwg, 0, w);
              phx = cmul(phx, lanczos_response(w, 0.5f));
            }
            const int e = NP * LS + l;
            const float2 pn = k_eig > 0 ? eigen_bin(psf_hat, PSF_ELEMS, k_eig, pc, e) : __ldg(psf_hat + e);
            nyb[l] = cmul(pn, cmul(phx, phy));
            if constexpr (LZ) {
              nybx[l] = cmul(pn, cmul(phxd, phy));
              nyby[l] = cmul(pn, cmul(phx, phyd));
            }
            nys[C::NYS * l + 0] = s;
            nys[C::NYS * l + 1] = sq;
            nys[C::NYS * l + 2] = sn;
            if constexpr (WN) nys[C::NYS * l + 3] = sd;
          }
        } else if (i < t3) {
          const int k = i - t2;
          float2 ph;
          sincospif(-2.0f * gx * (float)k * INV_N, &ph.y, &ph.x);
          if constexpr (LZ) {
            float w[7];
            load_weights(lwg, 8, w);
            pxd[k] = cmul(ph, lanczos_slope_response(w, (float)k * INV_N));
            load_weights(lwg, 0, w);
            ph = cmul(ph, lanczos_response(w, (float)k * INV_N));
          }
          px[k] = ph;
        } else {
          const int t = i - t3;
          if (t < nrt) adj_real_term(r, ps.mog, ps.k, N, t, &at, k_eig > 0 ? pc + 8 : nullptr);
          else if (t < nr2) adj_real_term_zero(t, &at);
          else adj_component_tables(r, t - nr2, s_fa, s_fc, s_fd);
        }
      }
      landed = mbar_wait(bar, parity);
      parity ^= 1u;
    }
    if (tid == 0) s_pos = pos2;
    async_copy_wait();
    if (__syncthreads_or(!landed)) {
      if (tid == 0) set_status(p.status, MOG_ERR_TIMEOUT);
      return;
    }
    pos2 = s_pos;
    if (!work) {
      __syncthreads();   // s_pos has been read
      pos = pos1;
      pos1 = pos2;
      b3 = b3n;
      continue;
    }

    float acc[7] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
    // ---- real-space terms ----
    // run i of the group's row pairs: pair i / 4, row i % 4 / 2 of it, half i % 2
    // of the row (LZ: the convolution reaches into other groups' rows, from the
    // caller's patch)
    adj_real_runs<N, WN, LZ>(
        at, nr2, 4 * ROUNDS,
        [&](int i, int& y, int& x) {
          const int pr = pair_of((i >> 2) * GROUPS + f), h = (i >> 1) & 1;
          y = pr + h * NP;
          x = 8 * (j + T * (i & 1));
          return reinterpret_cast<const float*>(Z + pr * RS) + h * N + x;
        },
        acc, r.s11, r.s12, r.s22, grad_out + r.off, N, s_lw);
    __syncwarp();   // the group's rows have been read

    // ---- forward FFT of row pairs, packed as g[p] + i g[p + N/2] ----
    float2 v[16];
#pragma unroll 1
    for (int rr = 0; rr < ROUNDS; ++rr) {
      float2* const zr = Z + pair_of(rr * GROUPS + f) * RS;
      const float* g = reinterpret_cast<const float*>(zr) + j;
#pragma unroll
      for (int m = 0; m < 16; ++m) v[m] = make_float2(g[m * T], g[N + m * T]);
      __syncwarp();
      fft16<N, -1>(
          tw, v, [&](int k1) { return zr + k1 * T + (j ^ (k1 & (T - 1))); },
          [&](int q, int i) { return zr + (j + T * q) * T + (j ^ i); });
#pragma unroll
      for (int q = 0; q < 16 / T; ++q)
#pragma unroll
        for (int k2 = 0; k2 < T; ++k2) zr[j + T * q + 16 * k2] = v[fft16_at<N>(q, k2)];
    }
    __syncthreads();   // every row pair's spectrum is there

    // ---- columns, contraction ----
#pragma unroll 1
    for (int cc = 0; cc < ROUNDS; ++cc) {
      const int col = cc * GROUPS + f;   // column nu = col / N (column 0: nu = 0 and 1/2 packed)
      float2* const zk = Z + col;
      float2* const zm = Z + (col ? N - col : NP);
      // rows p and p + N/2, p = j + m T, have spectra (Z[k] + conj Z[N-k]) / 2 and
      // (Z[k] - conj Z[N-k]) / (2i); their nu = 0 and nu = 1/2 values are real,
      // packed as re + i im
#pragma unroll
      for (int m = 0; m < 8; ++m) {
        const float2 a = zk[(j + m * T) * RS], b = zm[(j + m * T) * RS];
        v[m] = col ? make_float2(0.5f * (a.x + b.x), 0.5f * (a.y - b.y)) : make_float2(a.x, b.x);
        v[m + 8] = col ? make_float2(0.5f * (a.y + b.y), -0.5f * (a.x - b.x)) : make_float2(a.y, b.y);
      }
      __syncwarp();
      fft16<N, -1>(
          tw, v,
          [&](int k1) { return ((k1 & 8) ? zm : zk) + ((k1 & 7) * T + (j ^ (k1 & (T - 1)))) * RS; },
          [&](int q, int i) { return (((T * q) & 8) ? zm : zk) + ((j + ((T * q) & 7)) * T + (j ^ i)) * RS; });
      if (col == 0) {   // packed U[l], l < N/2 at row l of zk, the others of zm
#pragma unroll
        for (int q = 0; q < 16 / T; ++q)
#pragma unroll
          for (int k2 = 0; k2 < T; ++k2)
            (k2 < T / 2 ? zk : zm)[(j + T * q + 16 * (k2 % (T / 2))) * RS] = v[fft16_at<N>(q, k2)];
      }
      __syncwarp();
      const float nu = col * INV_N, ck = col == 0 ? 1.0f : 2.0f;
      const float s11 = r.s11, s12x2 = 2.0f * r.s12, s22 = r.s22;
      const float a0 = s11 * nu * nu, a1 = s12x2 * nu, omj = (float)j * INV_N;
      const int nf = r.nf;
      const float2 pxk = px[col];
      [[maybe_unused]] const float2 pxdk = LZ ? pxd[col] : pxk;
      const float2* const pk = psf_hat + col * LS + j;
      // bins per sweep over the components (the registers of the Sersic sums
      // leave room for four)
      constexpr int BH = WN ? 4 : 8;
      // bin b < 16: hb = b / 8 (omega < 0), then q, k2 in turn: l = j + l_of(b)
      auto q_of = [](int b) { return (b & 7) / (T / 2); };
      auto k2_of = [](int b) { return (b & 7) % (T / 2) + (b >> 3) * (T / 2); };
#pragma unroll
      for (int b0 = 0; b0 < 16; b0 += BH) {
        const int hb = b0 >> 3;
        float2 qp[BH / 2], S[BH / 2], SQ[BH / 2], SN[BH / 2], SD[BH / 2];
#pragma unroll
        for (int i = 0; i < BH / 2; ++i) {
          const int la = T * q_of(b0 + 2 * i) + 16 * k2_of(b0 + 2 * i);
          const int lb = T * q_of(b0 + 2 * i + 1) + 16 * k2_of(b0 + 2 * i + 1);
          const float oa = omj + (float)(la - hb * N) * INV_N, ob = omj + (float)(lb - hb * N) * INV_N;
          qp[i] = make_float2(fmaf(oa, fmaf(s22, oa, a1), a0), fmaf(ob, fmaf(s22, ob, a1), a0));
        }
        adj_mixture_sums<BH / 2, WN>(s_fa, s_fc, s_fd, nf, qp, S, SQ, SN, SD);
        [[maybe_unused]] float2 pe[BH];
        if constexpr (EIG)
          if (k_eig > 0)
            eigen_bins(pk, PSF_ELEMS, k_eig, pc, [&](int i) { return T * q_of(b0 + i) + 16 * k2_of(b0 + i); }, pe);
#pragma unroll
        for (int i = 0; i < BH; ++i) {
          const int lo = T * q_of(b0 + i) + 16 * k2_of(b0 + i), l = j + lo;
          const float om = omj + (float)(lo - hb * N) * INV_N;
          float2 gk = v[fft16_at<N>(q_of(b0 + i), k2_of(b0 + i))];
          float2 gn = make_float2(0.f, 0.f);
          if (col == 0) {
            const int ln = (N - l) & (N - 1);
            const float2 u = (hb ? zm : zk)[(l & (NP - 1)) * RS], un = (ln >= NP ? zm : zk)[(ln & (NP - 1)) * RS];
            gk = make_float2(0.5f * (u.x + un.x), 0.5f * (u.y - un.y));
            gn = make_float2(0.5f * (u.y + un.y), -0.5f * (u.x - un.x));
          }
          const float s = (i & 1) ? S[i >> 1].y : S[i >> 1].x;
          const float sq = (i & 1) ? SQ[i >> 1].y : SQ[i >> 1].x;
          const float sn = (i & 1) ? SN[i >> 1].y : SN[i >> 1].x;
          const float sd = (i & 1) ? SD[i >> 1].y : SD[i >> 1].x;
          const float2 pv = (EIG && k_eig > 0) ? pe[i] : __ldg(pk + lo);
          float2 z;   // c_k conj(G) P phase
          if constexpr (LZ) {
            z = contract_shift(pv, gk, ck, pxk, pxdk, py[l], pyd[l], s, acc);
            contract_shape(z.x, nu, om, s, sq, sn, acc);
          } else {
            z = cscale(cmulc(cmul(pv, cmul(pxk, py[l])), gk), ck);
            contract_bin(z, nu, om, s, sq, sn, acc);
          }
          if constexpr (WN) acc[6] = fmaf(z.x, sd, acc[6]);
          if (col == 0) {
            const float2 zh = cmulc(nyb[l], gn);
            const float* const ny = nys + C::NYS * l;
            if constexpr (LZ) {
              acc[1] = fmaf(fmaf(nybx[l].x, gn.x, nybx[l].y * gn.y), ny[0], acc[1]);
              acc[2] = fmaf(fmaf(nyby[l].x, gn.x, nyby[l].y * gn.y), ny[0], acc[2]);
              contract_shape(zh.x, 0.5f, om, ny[0], ny[1], ny[2], acc);
            } else {
              contract_bin(zh, 0.5f, om, ny[0], ny[1], ny[2], acc);
            }
            if constexpr (WN) acc[6] = fmaf(zh.x, ny[3], acc[6]);
          }
        }
      }
    }

    // ---- reduce the sums over the CTA and apply the chain rule ----
#pragma unroll
    for (int k = 0; k < NACC; ++k) {
      float x = acc[k];
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
      if ((tid & 31) == 0) red[(tid >> 5) * 8 + k] = x;
    }
    __syncthreads();
    if (tid == 0) {
      float t[7] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
      for (int w = 0; w < WARPS; ++w)
        for (int k = 0; k < NACC; ++k) t[k] += red[w * 8 + k];
      float* out = grad_params + r.gal * NACC;
      if constexpr (WN) out[6] = t[6];
      out[0] = t[0] / r.flux;
      out[1] = (LZ ? 1.0f : TWO_PI) * t[1];
      out[2] = (LZ ? 1.0f : TWO_PI) * t[2];
#pragma unroll
      for (int k = 0; k < 3; ++k) out[3 + k] = t[3] * r.dS[k][0] + t[4] * r.dS[k][1] + t[5] * r.dS[k][2];
    }
    pos = pos1;
    pos1 = pos2;
    b3 = b3n;
  }
}

template <bool WN, bool EIG, bool LZ>
int bwd128_occupancy() {
  const int occ = kernel_occupancy(reinterpret_cast<const void*>(render_bwd128_kernel<WN, EIG, LZ>), THREADS,
                                   BCfg<WN, LZ>::SMEM);
  return occ < 0 ? occ : (occ < CTAS_PER_SM ? occ : CTAS_PER_SM);
}

template <bool WN, bool EIG, bool LZ>
cudaError_t launch_mode(const RenderParams& p, const float* grad_out, float* grad_params, int num_sms, int ctas_per_sm,
                        cudaStream_t s) {
  const int occ = bwd128_occupancy<WN, EIG, LZ>();
  if (occ < 0) return cudaErrorInvalidConfiguration;
  const int ctas = (ctas_per_sm > 0 && ctas_per_sm < occ) ? ctas_per_sm : occ;
  render_bwd128_kernel<WN, EIG, LZ>
      <<<persistent_grid(p, ctas, num_sms), THREADS, BCfg<WN, LZ>::SMEM, s>>>(p, grad_out, grad_params);
  return cudaGetLastError();
}

template <bool LZ>
cudaError_t launch_shift(const RenderParams& p, const float* grad_out, float* grad_params, int num_sms, int ctas_per_sm,
                         cudaStream_t s) {
  if (p.eigen)
    return p.grad_n ? launch_mode<true, true, LZ>(p, grad_out, grad_params, num_sms, ctas_per_sm, s)
                    : launch_mode<false, true, LZ>(p, grad_out, grad_params, num_sms, ctas_per_sm, s);
  return p.grad_n ? launch_mode<true, false, LZ>(p, grad_out, grad_params, num_sms, ctas_per_sm, s)
                  : launch_mode<false, false, LZ>(p, grad_out, grad_params, num_sms, ctas_per_sm, s);
}

}  // namespace

cudaError_t launch_render_bwd128(const RenderParams& p, const float* grad_out, float* grad_params, int num_sms,
                                 int ctas_per_sm, cudaStream_t s) {
  return p.lanczos ? launch_shift<true>(p, grad_out, grad_params, num_sms, ctas_per_sm, s)
                   : launch_shift<false>(p, grad_out, grad_params, num_sms, ctas_per_sm, s);
}

int render_bwd128_max_ctas() { return bwd128_occupancy<false, false, false>(); }

}  // namespace mog
