// Fused adjoint for 256 x 256 patches (gradients w.r.t. flux, x, y, log r_e,
// e1, e2 and optionally the Sersic index; the contraction of render_bwd.cu, see
// its header), 16 values per thread (fft16.cuh), a 512-thread CTA per SM, one
// galaxy at a time, 16 threads per transform, in two teams of 256 threads.
//
// Neither the gradient patch (256 KB) nor the half spectrum of its rows fits
// one CTA's shared memory, so the rows' spectra go through a per-CTA scratch in
// global memory (256 KB, [k][row pair], L2-resident where it can be):
//   rows      4 rounds per team of 16 row-pair forward FFTs, row pair (p, p + N/2)
//             packed as g[p] + i g[p + N/2].  First pass: 16 threads per row
//             pair, exchange through shared memory (two buffers and one barrier
//             of the team per round).  Second pass: 16 row pairs side by side per
//             half-warp, so that the outputs are stored as 128-byte segments
//             directly
//   parts     the four parts of bwd256.cuh, two per team, each
//     real      analytic real-space derivatives over its runs of pixels
//     columns   2 rounds of 16 columns: gather of elements k and N - k of every
//               row pair, untangled into the rows' spectra, forward FFT along
//               y, contraction with the mixture's derivatives
//     reduce    warp shuffles; after the last one thread applies the chain rule
// The PSF spectrum is read from global memory.  The operations and the order of
// the sums are those of the cluster kernel (render_bwd256c.cu), so a galaxy has
// the same gradients from both.
//
// Against 8 values per thread (radix 8 x 8 x 4, two exchanges per transform, the
// rows untangled through shared memory between two CTA barriers in each of 8
// rounds, two 512-thread CTAs at 64 registers; other sums than the clusters'):
// calls of 10.6k galaxies 3.10 -> 2.84 ms, with the Sersic index 3.73 -> 3.45,
// Lanczos 4.70 -> 4.02; of 304 0.222 -> 0.147.  Two 256-thread CTAs per SM, a
// galaxy each, take 2.76 for the 10.6k but 0.183 for the 304, and 126 us instead
// of 87 for 152.
#include "bwd256.cuh"

namespace mog {

namespace {

using namespace bwd256;

constexpr int TEAMS = 2;                  // of THREADS threads
constexpr int CTA_THREADS = TEAMS * THREADS;
constexpr int ROW_ROUNDS = NP / GROUPS;   // 8
// Exchange rows 273 float2 apart: odd, for the second pass that reads 16 row
// pairs side by side.
constexpr int CS = 16 * EX + 1;

template <bool LZ>
struct BCfg256 {
  static constexpr size_t off_w = 0;                                      // two buffers of 16 exchange rows per team
  static constexpr size_t off_py = off_w + 2 * TEAMS * sizeof(float2) * GROUPS * CS;
  static constexpr size_t off_px = off_py + sizeof(float2) * N;
  static constexpr size_t off_nb = off_px + sizeof(float2) * NP;
  static constexpr size_t off_ns = off_nb + sizeof(float2) * N;
  static constexpr size_t off_lz = off_ns + sizeof(float) * 4 * N;        // pyd, nybx, nyby, pxd
  static constexpr size_t off_rec = off_lz + (LZ ? sizeof(float2) * (3 * N + NP) : 0);
  static constexpr size_t off_terms = off_rec + 2 * sizeof(AdjRecord);
  static constexpr size_t off_red = off_terms + sizeof(AdjTerms);
  static constexpr size_t off_bar = off_red + sizeof(float) * 8 * PARTS * WARPS;
  static constexpr size_t SMEM = off_bar + 2 * sizeof(uint64_t);
  static_assert(off_rec % 16 == 0 && off_bar % 8 == 0, "alignment");
  static_assert(SMEM + 1024 <= 227 * 1024, "shared memory of a CTA");
};

// WN: also d L / d(Sersic n), a seventh gradient per galaxy.  EIG: some PSF of
// the context is an eigen-PSF (its spectrum combined bin by bin where read).
// LZ: the gradient of the Lanczos variant's model (see render_bwd.cu).
template <bool WN, bool EIG, bool LZ>
__global__ void __launch_bounds__(CTA_THREADS, 1)
    render_bwd256_kernel(RenderParams p, const float* __restrict__ grad_out, float* __restrict__ grad_params,
                         float2* __restrict__ scratch_all) {
  using C = BCfg256<LZ>;
  constexpr int NACC = WN ? 7 : 6;
  extern __shared__ __align__(128) unsigned char smem[];
  __shared__ float4 s_fa[KMAX], s_fc[KMAX], s_fd[KMAX];
  __shared__ float s_lw[LZ ? ADJ_LW : 1];
  __shared__ int s_pos[2];
  float2* W = reinterpret_cast<float2*>(smem + C::off_w);
  AdjRecord* rec = reinterpret_cast<AdjRecord*>(smem + C::off_rec);
  float* red = reinterpret_cast<float*>(smem + C::off_red);   // [part][warp][8]
  uint64_t* bar = reinterpret_cast<uint64_t*>(smem + C::off_bar);
  float2* const lz = reinterpret_cast<float2*>(smem + C::off_lz);
  Tables t;
  t.py = reinterpret_cast<float2*>(smem + C::off_py);
  t.px = reinterpret_cast<float2*>(smem + C::off_px);
  t.nyb = reinterpret_cast<float2*>(smem + C::off_nb);
  t.nys = reinterpret_cast<float*>(smem + C::off_ns);
  t.pyd = lz;
  t.nybx = lz + N;
  t.nyby = lz + 2 * N;
  t.pxd = lz + 3 * N;
  t.at = reinterpret_cast<AdjTerms*>(smem + C::off_terms);
  t.fa = s_fa;
  t.fc = s_fc;
  t.fd = s_fd;
  t.lw = s_lw;

  const int tid = threadIdx.x;
  const int team = tid / THREADS, tt = tid % THREADS;
  const int f = tt / T, j = tt % T;
  float2* const scratch = scratch_all + (size_t)blockIdx.x * N * NP;   // [k][row pair]
  float2 tw[15];
  fft16_twiddles<N>(j, tw);
  const int count = p.bucket_count[B], first = p.bucket_start[B];
  if (count < p.bucket_min || count > p.bucket_max) return;   // the other kernel's (launch_by_count)
  const unsigned char* records = p.records + (size_t)first * sizeof(AdjRecord);
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
  if (tid == 0) {
    mbar_init(&bar[0], 1);
    mbar_init(&bar[1], 1);
    q_ahead = atomicAdd(&p.queue[B], p.chunk);
    const int p0 = next_position();
    s_pos[0] = p0;
    if (p0 >= 0) bulk_load(&rec[0], records + (size_t)p0 * sizeof(AdjRecord), sizeof(AdjRecord), &bar[0]);
  }
  uint32_t rec_parity = 0;

  // No barrier at the top of the loop: the previous galaxy's last one (the
  // sums) follows every read of its tables, work rows and scratch; after it
  // only thread 0 reads (the sums, and the record, whose buffer it refills
  // itself later).
  __syncthreads();
  for (int buf = 0;; buf ^= 1) {
    const int pos = s_pos[buf];
    if (pos < 0) break;
    if (tid == 0) {
      const int np = next_position();
      s_pos[buf ^ 1] = np;
      if (np >= 0)
        bulk_load(&rec[buf ^ 1], records + (size_t)np * sizeof(AdjRecord), sizeof(AdjRecord), &bar[buf ^ 1]);
    }
    const bool landed = mbar_wait(&bar[buf], (rec_parity >> buf) & 1u);
    rec_parity ^= 1u << buf;
    const AdjRecord& r = rec[buf];
    const bool work = landed && r.ok != 0;   // read before the barrier: a skipped galaxy's record may be replaced after it
    if (__syncthreads_or(!landed)) {
      if (tid == 0) set_status(p.status, MOG_ERR_TIMEOUT);
      return;
    }
    if (!work) continue;   // uniform
    const DevPsf& ps = p.psfs[r.psf];
    const float* pc = p.pcoef + ((size_t)first + pos) * PCOEF;
    const int k_eig = EIG ? ps.k_eig : 0;
    const float2* const psf_hat = ps.spec[B];
    const float* gpatch = grad_out + r.off;
    const int nr2 = real_terms_padded(r.nrc * ps.k);
    make_tables<WN, EIG, LZ>(t, r, ps, pc, LZ ? p.lzw + ((size_t)first + pos) * ADJ_LW : nullptr, 0, NP, true, tid,
                             CTA_THREADS);

    // ---- rows ----
    float2 v[16];
#pragma unroll 1
    for (int i = 0; i < ROW_ROUNDS / TEAMS; ++i) {
      const int rr = i * TEAMS + team;
      const float* ga = gpatch + (size_t)(GROUPS * rr + f) * N + j;
      const float* gb = ga + (N / 2) * N;
#pragma unroll
      for (int m = 0; m < 16; ++m) v[m] = make_float2(__ldg(ga + m * T), __ldg(gb + m * T));
      float2* const wb = W + ((i & 1) * TEAMS + team) * GROUPS * CS;
      dft16<-1>(v);
#pragma unroll
      for (int k1 = 0; k1 < 16; ++k1) wb[f * CS + k1 * EX + j] = k1 ? cmulc(v[at16(k1)], tw[k1 - 1]) : v[0];
      // this round's first passes are done (and the reads of the round before last)
      asm volatile("bar.sync %0, %1;" ::"r"(1 + team), "n"(THREADS) : "memory");
      // second pass: thread (k1, c) of row pair 16 rr + c, c along the half-warp
      const float2* const rd = wb + j * CS + f * EX;
#pragma unroll
      for (int u = 0; u < 16; ++u) v[u] = rd[u];
      dft16<-1>(v);
      float2* const z = scratch + f * NP + GROUPS * rr + j;
#pragma unroll
      for (int k2 = 0; k2 < 16; ++k2) z[16 * k2 * NP] = v[at16(k2)];
    }
    __syncthreads();   // tables and scratch complete and visible; W is free

    // ---- the parts: real-space terms, columns, sums ----
    float2* const w = W + (team * GROUPS + f) * CS;
#pragma unroll 1
    for (int part = team; part < PARTS; part += TEAMS) {
      float acc[7] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
      adj_real_space<N, WN, LZ>(gpatch, N, *t.at, nr2, part * THREADS + tt, PARTS * THREADS, acc, r.s11, r.s12, r.s22,
                                s_lw);
#pragma unroll 1
      for (int cc = 0; cc < ROUNDS; ++cc) {
        const int k = part * KL + cc * GROUPS + f;   // column nu = k / N (column 0: nu = 0 and 1/2 packed)
        const float2* const zk = scratch + (size_t)k * NP + j;
        const float2* const zn = scratch + (size_t)(k ? N - k : N / 2) * NP + j;
#pragma unroll
        for (int m = 0; m < 8; ++m) untangle(k, __ldcg(zk + 16 * m), __ldcg(zn + 16 * m), v[m], v[m + 8]);
        // (the registers of the Sersic sums leave room for four bins at a time)
        column<WN ? 4 : 8, WN, EIG, LZ>(t, r, psf_hat, k_eig, pc, k, t.px[k], LZ ? t.pxd[k] : make_float2(0.f, 0.f), tw,
                                        v, w, j, acc);
      }
#pragma unroll
      for (int c = 0; c < NACC; ++c) {
        const float x = warp_sum(acc[c]);
        if ((tt & 31) == 0) red[(part * WARPS + (tt >> 5)) * 8 + c] = x;
      }
    }
    __syncthreads();   // the sums are there
    if (tid == 0) write_gradients<WN, LZ>(r, red, grad_params);
  }
}

}  // namespace

// One N/2 x N slice per CTA: the forward kernel (adding to patches) runs two CTAs
// per SM, the adjoint one.
size_t render_bwd256_scratch_bytes(int num_sms) {
  return sizeof(float2) * (size_t)2 * num_sms * (N / 2) * N;
}

static cudaError_t launch_many(const RenderParams& p, const float* grad_out, float* grad_params, float2* scratch,
                               int num_sms, cudaStream_t s) {
  auto fn = p.lanczos ? (p.eigen ? (p.grad_n ? render_bwd256_kernel<true, true, true> : render_bwd256_kernel<false, true, true>)
                                 : (p.grad_n ? render_bwd256_kernel<true, false, true> : render_bwd256_kernel<false, false, true>))
                      : (p.eigen ? (p.grad_n ? render_bwd256_kernel<true, true, false> : render_bwd256_kernel<false, true, false>)
                                 : (p.grad_n ? render_bwd256_kernel<true, false, false> : render_bwd256_kernel<false, false, false>));
  const size_t smem = p.lanczos ? BCfg256<true>::SMEM : BCfg256<false>::SMEM;
  if (kernel_occupancy(reinterpret_cast<const void*>(fn), CTA_THREADS, smem) < 0) return cudaErrorInvalidConfiguration;
  fn<<<persistent_grid(p, 1, num_sms), CTA_THREADS, smem, s>>>(p, grad_out, grad_params, scratch);
  return cudaGetLastError();
}

// Few galaxies: a cluster per galaxy (render_bwd256c.cu).  Up to one galaxy per SM
// the call takes as long as one CTA for one, 85 to 100 us (Lanczos 120 to 150); the
// clusters, 38 at a time, take 23 us (31) for each 38.  Calls on clusters and on
// this kernel, 114 galaxies: 93 and 101 us (with the Sersic index 105 and 111), 152:
// 115 and 87; Lanczos, 228: 206 and 211, 266: 233 and 226.
cudaError_t launch_render_bwd256(const RenderParams& p, const float* grad_out, float* grad_params, float2* scratch,
                                 int num_sms, cudaStream_t s, const SideStream* side) {
  return launch_by_count(
      p, few256_adjoint(p.lanczos != 0, num_sms), far256_adjoint(num_sms), s, side,
      [&](const RenderParams& q, cudaStream_t qs) {
        return launch_render_bwd256_small(q, grad_out, grad_params, num_sms, qs);
      },
      [&](const RenderParams& q, cudaStream_t qs) {
        return launch_many(q, grad_out, grad_params, scratch, num_sms, qs);
      });
}

}  // namespace mog
