// Adjoint of 256 x 256 patches for small batches (gradients w.r.t. flux, x, y,
// log r_e, e1, e2 and optionally the Sersic index; the contraction of
// render_bwd.cu, see its header): one galaxy at a time per cluster of four
// 256-thread CTAs, 16 values per thread (fft16.cuh).  A CTA of
// render_bwd256.cu takes 85 to 100 us for a galaxy, whatever the batch; when
// there are fewer galaxies than SMs, spreading one over four SMs is what
// shortens the call (one galaxy 27 us, 40 44 against 85, 76 67 against 94).
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
#include "bwd256.cuh"
#include "cluster.cuh"

namespace mog {

namespace {

using namespace bwd256;

constexpr int CL = PARTS;               // CTAs per galaxy, a part each
constexpr int RS = 16 * EX;             // a group's work row
// Output k of the CTA's row pair pl at k SZ + pl: an odd stride for the 16 k
// that a half-warp writes; the 16 row pairs that it gathers lie side by side.
constexpr int SZ = KL + 1;

constexpr size_t off_z = 0;
constexpr size_t off_w = off_z + sizeof(float2) * N * SZ;
constexpr size_t off_py = off_w + sizeof(float2) * GROUPS * RS;
constexpr size_t off_px = off_py + sizeof(float2) * N;   // the CTA's columns
constexpr size_t off_nb = off_px + sizeof(float2) * KL;  // rank 0: nu = 1/2 column, P phase
constexpr size_t off_ns = off_nb + sizeof(float2) * N;   // and the mixture sums
constexpr size_t off_rec = (off_ns + sizeof(float) * 4 * N + 15) & ~size_t(15);
// LZ: phase times slope response along omega and nu; the nu = 1/2 column's P
// phase with the slopes along x and along y
constexpr size_t LZ_ELEMS = 3 * N + KL;
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
  constexpr int NACC = WN ? 7 : 6;
  extern __shared__ __align__(128) unsigned char smem[];
  __shared__ float4 s_fa[KMAX], s_fc[KMAX], s_fd[KMAX];
  __shared__ float s_lw[LZ ? ADJ_LW : 1];
  float2* Z = reinterpret_cast<float2*>(smem + off_z);
  float2* W = reinterpret_cast<float2*>(smem + off_w);
  AdjRecord* rec = reinterpret_cast<AdjRecord*>(smem + off_rec);
  float* red = reinterpret_cast<float*>(smem + off_red);   // rank 0: [CTA][warp][8]
  float2* const lz = reinterpret_cast<float2*>(smem + off_lz);
  Tables t;
  t.py = reinterpret_cast<float2*>(smem + off_py);
  t.px = reinterpret_cast<float2*>(smem + off_px);
  t.nyb = reinterpret_cast<float2*>(smem + off_nb);
  t.nys = reinterpret_cast<float*>(smem + off_ns);
  t.pyd = lz;
  t.nybx = lz + N;
  t.nyby = lz + 2 * N;
  t.pxd = lz + 3 * N;
  t.at = reinterpret_cast<AdjTerms*>(smem + off_terms);
  t.fa = s_fa;
  t.fc = s_fc;
  t.fd = s_fd;
  t.lw = s_lw;

  const int tid = threadIdx.x;
  const int f = tid / T, j = tid % T;
  const int rank = (int)cluster_rank();
  float2 tw[15];
  fft16_twiddles<N>(j, tw);
  float2* const w = W + f * RS;
  auto at_k1 = [&](int k1) { return w + k1 * EX + j; };
  auto at_i = [&](int, int i) { return w + j * EX + i; };
  const int count = p.bucket_count[B], first = p.bucket_start[B];
  if (count < p.bucket_min || count > p.bucket_max) return;   // the other kernel's (launch_by_count), for the whole cluster
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
    make_tables<WN, EIG, LZ>(t, r, ps, pc, LZ ? p.lzw + ((size_t)first + pos) * ADJ_LW : nullptr, rank * KL, KL,
                             rank == 0, tid, THREADS);
    __syncthreads();

    float acc[7] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
    adj_real_space<N, WN, LZ>(gpatch, N, *t.at, real_terms_padded(r.nrc * ps.k), rank * THREADS + tid, CL * THREADS, acc,
                              r.s11, r.s12, r.s22, s_lw);

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
      // row pair p = j + 16 m lies in CTA m / 2
      const uint32_t zk = smem_u32(Z + k * SZ + j), zn = smem_u32(Z + (k ? N - k : N / 2) * SZ + j);
#pragma unroll
      for (int m = 0; m < 8; ++m) {
        const float2 a = cluster_ld2(cluster_map(zk + 8 * 16 * (m & 1), m >> 1));
        const float2 b = cluster_ld2(cluster_map(zn + 8 * 16 * (m & 1), m >> 1));
        untangle(k, a, b, v[m], v[m + 8]);
      }
      column<8, WN, EIG, LZ>(t, r, psf_hat, k_eig, pc, k, t.px[cc * GROUPS + f],
                             LZ ? t.pxd[cc * GROUPS + f] : make_float2(0.f, 0.f), tw, v, w, j, acc);
    }

    // ---- reduce and chain rule ----
    const uint32_t slot = cluster_map(smem_u32(red + (rank * WARPS + (tid >> 5)) * 8), 0);
#pragma unroll
    for (int c = 0; c < NACC; ++c) {
      const float x = warp_sum(acc[c]);
      if ((tid & 31) == 0) cluster_st(slot + 4 * c, x);
    }
    sync_all();   // the sums are there, and every gather of Z has returned
    if (rank == 0 && tid == 0) write_gradients<WN, LZ>(r, red, grad_params);
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
