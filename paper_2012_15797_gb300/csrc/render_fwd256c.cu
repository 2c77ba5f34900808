// Forward render of 256 x 256 patches for small batches (Section 2, Steps
// 3-8): one galaxy at a time per cluster of four 256-thread CTAs, 16 values per
// thread (fft16.cuh).  A CTA of render_fwd256.cu takes about 80 us for a galaxy,
// whatever the batch; when there are fewer galaxies than CTAs fit, spreading one
// over four SMs is what shortens the call (one galaxy 65 -> 24 us, 100 98 -> 52,
// with the loss 108 -> 56, Lanczos 151 -> 83, composites 118 -> 71).
//
// The galaxy's N/2 packed columns (nu = 0 and nu = 1/2 share one) and its N/2
// row pairs (p, p + N/2) are spread evenly over the cluster's CTAs, 16 threads
// per transform, two rounds per direction:
//
//   columns   Fourier mixture x PSF spectrum (read from L2) x phase on the
//             thread's 16 bins, inverse transform along omega; the thread ends
//             with rows p and p + N/2 of its column, so it forms both elements
//             Z_p[k], Z_p[N - k] of their shared row transform and leaves them
//             in its own CTA's shared memory
//   rows      each thread gathers its row pair's 16 inputs from the CTAs that
//             hold the columns (distributed shared memory), inverse transform
//             along nu, real-space terms added, two pixel rows stored
//
// Per galaxy: one cluster barrier between the columns and the rows and one,
// split into arrive and wait, between the rows' gathers and the next galaxy's
// columns.  Those barriers and the gathers are what bounds it in a large batch
// (10.6k galaxies: 2.19 ms against 2.00 ms of render_fwd256.cu).
#include "cluster.cuh"
#include "fwd16.cuh"


namespace mog {

namespace {

constexpr int N = 256;
constexpr int T = fft16_threads<N>();   // threads per transform
constexpr int CL = 4;                   // CTAs per galaxy
constexpr int KL = N / 2 / CL;          // columns (and row pairs) per CTA
constexpr int THREADS = 256;
constexpr int GROUPS = THREADS / T;
constexpr int ROUNDS = KL / GROUPS;
constexpr int WARPS = THREADS / 32;
constexpr int CTAS_PER_SM = 2;
constexpr int LS = psf_lstride(N);
constexpr int PSF_ELEMS = psf_spec_elems(N);
constexpr int B = bucket_of(N);
constexpr int HALF = N / 2 + 2;         // omega = 0 .. 1/2 (padded)
// A group's work row: exchange element (k1, i) at 17 k1 + i (conflict free both
// ways), then the two pixel rows.
constexpr int EX = T + 1;
constexpr int RS = 16 * EX;
// Rows of the two spectra halves: slot kl of row p holds Z_p[k] (ZA) and
// Z_p[N - k] (ZM) of the CTA's column k = column(kl); Z_p[N/2] is in rank 0's
// ZM slot 0, which k = 0 leaves free.  The odd stride spreads the 16 rows that a
// half-warp writes, and its 16 gathered columns lie side by side.
constexpr int SZ = KL + 1;

// The columns are shared out in blocks of 16: rank c has block c, then block
// 7 - c, so that every CTA gets as many of the low frequencies (where no
// component is skipped) as the others, and the 16 inputs that a half-warp
// gathers with one load lie in one CTA side by side.
static_assert(GROUPS == 16 && ROUNDS == 2 && CL == 4, "blocks of 16 columns");
__device__ __forceinline__ int column(int kl, int rank) {
  return kl < 16 ? 16 * rank + kl : 16 * (7 - rank) + kl - 16;
}
__host__ __device__ __forceinline__ constexpr int block_rank(int b) { return b < 4 ? b : 7 - b; }
__host__ __device__ __forceinline__ constexpr int block_slot(int b) { return b < 4 ? 0 : 16; }

template <bool COMP>
struct CfgC {
  using RT = RealTermsN<COMP ? 2 * RMAX : RMAX>;
  static constexpr int RECS = COMP ? 2 : 1;   // records per galaxy
  static constexpr size_t off_za = 0;
  static constexpr size_t off_zm = off_za + sizeof(float2) * (N / 2) * SZ;
  static constexpr size_t off_w = off_zm + sizeof(float2) * (N / 2) * SZ;
  // per galaxy, two buffers: phases along omega and nu, the nu = 1/2 column,
  // Fourier components, real-space terms; records: three
  static constexpr size_t off_py = off_w + sizeof(float2) * GROUPS * RS;
  static constexpr size_t off_px = off_py + 2 * sizeof(float2) * HALF;
  static constexpr size_t off_hn = off_px + 2 * sizeof(float2) * KL;
  static constexpr size_t off_fc = (off_hn + 2 * sizeof(float2) * HALF + 15) & ~size_t(15);
  static constexpr size_t off_rec = off_fc + 2 * sizeof(float4) * RECS * KMAX;
  static constexpr size_t off_rt = off_rec + 3 * RECS * sizeof(GalaxyRecord);
  static constexpr size_t SMEM = off_rt + 2 * sizeof(RT);
  // Lanczos: the real-space rows, convolved along x, take the place of Z
  static_assert(sizeof(float) * KL * 2 * N <= off_w, "real-space rows");
  static_assert(CTAS_PER_SM * (SMEM + 144 + 1024) <= 228 * 1024, "two CTAs share an SM's shared memory");
};

// LZ: the Lanczos sub-pixel shift (records carry the integer offset and the
// fraction): the convolution of the Fourier part is folded into the phase
// tables, the real-space part is convolved along x in the group's own rows,
// then along y over the rows of all groups (and CTAs).  EIG: some PSF of the
// context is an eigen-PSF.  LOSS: the loss mode of mog_render_chi2.  COMP:
// composites of two profiles (p.records2).
template <bool LZ, bool EIG, bool LOSS, bool COMP>
__global__ void __launch_bounds__(THREADS, CTAS_PER_SM) render_fwd256c_kernel(RenderParams p) {
  using C = CfgC<COMP>;
  using RT = typename C::RT;
  static_assert(!(LZ && LOSS), "the loss mode renders with the phase shift");
  static_assert(!(COMP && (EIG || LOSS)), "composites: constant PSFs, plain render");
  constexpr float INV_N = 1.0f / N;
  extern __shared__ __align__(128) unsigned char smem[];
  float2* ZA = reinterpret_cast<float2*>(smem + C::off_za);
  float2* ZM = reinterpret_cast<float2*>(smem + C::off_zm);
  float2* W = reinterpret_cast<float2*>(smem + C::off_w);
  float2* pys = reinterpret_cast<float2*>(smem + C::off_py);   // [buffer][omega N = 0 .. N/2]
  float2* pxs = reinterpret_cast<float2*>(smem + C::off_px);   // [buffer][KL]
  float2* hns = reinterpret_cast<float2*>(smem + C::off_hn);   // [buffer][omega N = 0 .. N/2]
  float4* fcs = reinterpret_cast<float4*>(smem + C::off_fc);   // [buffer][RECS * KMAX]
  GalaxyRecord* rec = reinterpret_cast<GalaxyRecord*>(smem + C::off_rec);   // [3][RECS]
  RT* rts = reinterpret_cast<RT*>(smem + C::off_rt);
  __shared__ int s_first[3], s_pos[2];
  __shared__ float s_lzw[LZ ? 2 : 1][16];   // per buffer: Lanczos weights along x [0, 7) and y [8, 15)
  __shared__ float s_chi[LOSS ? 2 : 1][LOSS ? CL * WARPS : 1];   // rank 0: each warp's sum of squared residuals

  const int tid = threadIdx.x;
  const int f = tid / T, j = tid % T;
  const uint32_t rank = cluster_rank();
  const bool lead = rank == 0 && tid == 0;
  float2 tw[15];
  fft16_twiddles<N>(j, tw);
  float2* const w = W + f * RS;                 // the group's work row
  const int cx = (f & 1) * T;   // staged output rows, see below
  const int count = p.bucket_count[B];
  if (count < p.bucket_min || count > p.bucket_max) return;   // the other kernel's (launch_by_count), for the whole cluster
  const int first = p.bucket_start[B];          // planned position of this bucket's first galaxy
  const unsigned char* records = p.records + (size_t)first * RECORD_BYTES;
  [[maybe_unused]] const unsigned char* records2 = COMP ? p.records2 + (size_t)first * RECORD_BYTES : nullptr;

  // The work queue is taken by the lead thread, p.chunk positions at a time
  // with the next chunk requested one chunk ahead, and each position is
  // published to the cluster three galaxies ahead.
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
  auto publish = [&](int* slot, int v) {
    const uint32_t a = smem_u32(slot);
    for (int c = 0; c < CL; ++c) cluster_st(cluster_map(a, c), v);
  };
  auto sync_all = [&]() {
    cluster_arrive();
    cluster_wait();
  };
  // the record(s) of planned position pos into buffer b (16-byte pieces, one
  // per thread)
  auto load_records = [&](int b, int pos) {
    constexpr int PIECES = sizeof(GalaxyRecord) / 16;
    float4* const d = reinterpret_cast<float4*>(&rec[b * C::RECS]) + tid;
    if (tid < PIECES) async_copy16(d, reinterpret_cast<const float4*>(records + (size_t)pos * RECORD_BYTES) + tid);
    else if (COMP && tid < 2 * PIECES)
      async_copy16(d, reinterpret_cast<const float4*>(records2 + (size_t)pos * RECORD_BYTES) + tid - PIECES);
  };
  // LOSS, lead thread, once every warp has added its residuals of chi_gal
  long long chi_gal = -1;
  float chi_iv = 0.0f;
  int chi_buf = 0;
  auto write_chi2 = [&]() {
    if (chi_gal >= 0) {
      float t = 0.0f;
      for (int i = 0; i < CL * WARPS; ++i) t += s_chi[chi_buf][i];
      p.chi2[chi_gal] = chi_iv * t;
      chi_gal = -1;
    }
  };

  // Tables of a galaxy.  Phases and the nu = 1/2 column are kept for omega =
  // 0 .. 1/2: at -omega they are the complex conjugates (also the Lanczos
  // responses, whose weights are real).  hn: the Hermitian part of the nu =
  // 1/2 column, the mean of its value at omega and the conjugate at -omega,
  // for the CTA of column 0.
  auto shift_phase = [&](float g, float fr, const float* lzw) {
    float2 ph;
    sincospif(-2.0f * g * fr, &ph.y, &ph.x);
    if constexpr (LZ) {
      float wv[7];
      load_weights(lzw, 0, wv);
      ph = cmul(ph, lanczos_response(wv, fr));
    }
    return ph;
  };
  auto fourier_tables = [&](int b, const GalaxyRecord* r, int pos) {
    if (!r->ok) return;
    const DevPsf& ps = p.psfs[r->psf];
    const float2* const spec = ps.spec[B];
    const int k_eig = EIG ? ps.k_eig : 0;
    const float* pc = p.pcoef + ((size_t)first + pos) * PCOEF;
    const float* lzw = LZ ? p.lzw + ((size_t)first + pos) * 16 : nullptr;
    const float gx = r->x, gy = r->y;
    const int nf1 = r->nf, nfa = nf1 + (COMP ? r[1].nf : 0);
    constexpr int NH = N / 2 + 1;
    const int t1 = NH + KL, t2 = t1 + nfa, t3 = t2 + (rank == 0 ? NH : 0);
    for (int i = tid; i < t3; i += THREADS) {
      if (i < NH) {
        pys[b * HALF + i] = shift_phase(gy, (float)i * INV_N, LZ ? lzw + 8 : nullptr);
      } else if (i < t1) {
        pxs[b * KL + i - NH] = shift_phase(gx, (float)column(i - NH, rank) * INV_N, lzw);
      } else if (i < t2) {
        const int c = i - t1;
        const GalaxyRecord& rr = r[(COMP && c >= nf1) ? 1 : 0];
        const int cc = c - (COMP && c >= nf1 ? nf1 : 0);
        fcs[b * C::RECS * KMAX + c] = make_float4(rr.famp[cc], rr.famp[cc], rr.fcoef[cc], rr.fcoef[cc]);
      } else {
        const int l = i - t2;
        const float om = (float)l * INV_N;
        float2 val[2];
        const float2 phx = shift_phase(gx, 0.5f, lzw), phy = shift_phase(gy, om, LZ ? lzw + 8 : nullptr);
#pragma unroll
        for (int h = 0; h < 2; ++h) {   // at omega and -omega; N/2 is one bin, omega = -1/2
          const float o = (h || l == N / 2) ? -om : om;
          float acc = 0.0f;
#pragma unroll
          for (int u = 0; u < C::RECS; ++u) {
            const GalaxyRecord& rr = r[u];
            const float q = fmaf(o, fmaf(rr.s22, o, rr.s12), 0.25f * rr.s11);
            for (int c = 0; c < rr.nf; ++c) acc = fmaf(rr.famp[c], ex2(rr.fcoef[c] * q), acc);
          }
          const int e = (N / 2) * LS + (h ? (N - l) & (N - 1) : l);
          const float2 pn = (EIG && k_eig) ? eigen_bin(spec, PSF_ELEMS, k_eig, pc, e) : __ldg(spec + e);
          val[h] = cscale(cmul(pn, cmul(phx, (h || l == N / 2) ? conjf2(phy) : phy)), acc);
        }
        hns[b * HALF + l] = make_float2(0.5f * (val[0].x + val[1].x), 0.5f * (val[0].y - val[1].y));
      }
    }
  };

  sync_all();   // every CTA of the cluster runs: its shared memory may be written
  if (lead) {
    q_ahead = atomicAdd(&p.queue[B], p.chunk);
    for (int i = 0; i < 3; ++i) publish(&s_first[i], next_position());
  }
  sync_all();
  int pos = s_first[0], pos1 = s_first[1], pos2 = s_first[2];
  if (pos >= 0) load_records(0, pos);
  if (pos1 >= 0) load_records(1, pos1);
  async_copy_wait();
  __syncthreads();
  if (pos >= 0) fourier_tables(0, rec, pos);
  __syncthreads();

  // Who waits for whom.  Per galaxy i the cluster meets once (C1(i)), between
  // its columns and its rows, and once more in two parts (C2(i)): arrival when
  // the rows' gathers have returned, wait before Z of i + 1 is written.
  // Before C1(i): the columns of i (reading its Fourier tables and record),
  // the Fourier tables of i + 1 (buffer (i + 1) & 1, last read before
  // C1(i - 1); from the record of i + 1, loaded before C1(i - 1)), the
  // real-space terms of i (buffer i & 1, last read by the rows of i - 2) and
  // the record of i + 2 (the buffer of i - 1, last read before C1(i - 1)).
  // The rows use no record: what they need of it is in registers.
  bool pending = false;   // an arrival at C2 whose wait is still to come
  int b3 = 0;
  for (int buf = 0; pos >= 0; buf ^= 1) {
    const GalaxyRecord* const r = rec + b3 * C::RECS;
    const int b3n = b3 == 2 ? 0 : b3 + 1;
    const bool work = r->ok != 0;   // uniform over the cluster: every CTA reads the same record
    RT& rt = rts[buf];
    const float* pc = p.pcoef + ((size_t)first + pos) * PCOEF;
    const DevPsf& ps = p.psfs[work ? r->psf : 0];
    const float2* const psf_hat = ps.spec[B];
    const int k_eig = EIG ? ps.k_eig : 0;
    const int kp = ps.k, nrt1 = work ? r->nrc * kp : 0, nrt = nrt1 + (COMP && work ? r[1].nrc * kp : 0);
    const int nr = real_terms_padded(nrt);
    const int64_t off = r->off;
    [[maybe_unused]] const int64_t gal = r->gal;
    if (pos2 >= 0) load_records(b3n == 2 ? 0 : b3n + 1, pos2);
    int pos3 = -1;
    if (lead) pos3 = next_position();
    [[maybe_unused]] const float* const dat = (LOSS && work) ? (p.dptr ? p.dptr[gal] : p.data + off) : nullptr;
    if constexpr (LOSS) {
      // the data rows that this CTA's stores read, on their way to L2
      if (work)
        for (int i = tid; i < KL * N / 16; i += THREADS) {
          const int h = i / (KL * N / 32), o = i % (KL * N / 32);
          prefetch_l2(dat + (size_t)(h * (N / 2) + rank * KL) * N + 32 * o);
        }
    }

    // ---- Steps 5-6 on the bins l = j + m T of each of the group's columns, Step 7a ----
    float2 v[16];
    if (work) {
      const float2* const py = pys + buf * HALF;
      const float4* const fc = fcs + buf * C::RECS * KMAX;
#pragma unroll 1
      for (int cc = 0; cc < ROUNDS; ++cc) {
        // column nu = col / N; the second round from the far end of the block
        const int kl = cc ? KL - 1 - f : f, col = column(kl, rank);
        const float2* ph = psf_hat + col * LS + j;
        if (EIG && k_eig) {
          eigen_bins(ph, PSF_ELEMS, k_eig, pc, [](int m) { return m * T; }, v);
        } else {
#pragma unroll
          for (int m = 0; m < 16; ++m) v[m] = __ldg(ph + m * T);
        }
        float2 s[8];
#pragma unroll
        for (int k = 0; k < 8; ++k) s[k] = make_float2(0.0f, 0.0f);
        const float nu = (float)col * INV_N, omj = (float)j * INV_N;
        mixture16(fc, r->nf, r->s11, 2.0f * r->s12, r->s22, nu, omj, s);
        if constexpr (COMP) {
          mixture16(fc + r->nf, r[1].nf, r[1].s11, 2.0f * r[1].s12, r[1].s22, nu, omj, s);
        }
        const float2 pxk = pxs[buf * KL + kl];
#pragma unroll
        for (int m = 0; m < 16; ++m) {
          const int l = j + m * T;
          const float2 ph = m < 8 ? cmul(pxk, py[l]) : cmulc(pxk, py[N - l]);
          v[m] = cscale(cmul(v[m], ph), (m & 1) ? s[m >> 1].y : s[m >> 1].x);
        }
        if (col == 0) {
          // Pack the Hermitian parts of the nu = 0 and nu = 1/2 columns as
          // re + i im.  The nu = 0 column is Hermitian in omega by construction
          // (its self-conjugate bin l = N/2 keeps its real part).
          const float2* const hn = hns + buf * HALF;
#pragma unroll
          for (int m = 0; m < 16; ++m) {
            const int l = j + m * T;
            const float2 dc = (l == N / 2) ? make_float2(v[m].x, 0.0f) : v[m];
            const float2 h = m < 8 ? hn[l] : conjf2(hn[N - l]);
            v[m] = make_float2(dc.x - h.y, dc.y + h.x);
          }
        }
        fft16<N, +1>(
            tw, v, [&](int k1) { return w + k1 * EX + j; }, [&](int q, int i) { return w + j * EX + i; });
        if (pending) {   // C2 of the previous galaxy
          cluster_wait();
          pending = false;
        }
        // rows n = j + T q + 16 k2 of the column: pairs (p, p + N/2) are k2, k2 + T/2
        float2* za = ZA + j * SZ + kl;
        float2* zm = ZM + j * SZ + kl;
#pragma unroll
          for (int k2 = 0; k2 < T / 2; ++k2) {
            const float2 A = v[fft16_at<N>(0, k2)], Bv = v[fft16_at<N>(0, k2 + T / 2)];
            const int o = 16 * k2 * SZ;
            if (col > 0) {
              za[o] = make_float2(A.x - Bv.y, A.y + Bv.x);
              zm[o] = make_float2(A.x + Bv.y, Bv.x - A.y);
            } else {   // Z_p[0] and Z_p[N/2]
              za[o] = make_float2(A.x, Bv.x);
              zm[o] = make_float2(A.y, Bv.y);
            }
          }
      }
    } else if (pending) {
      cluster_wait();
      pending = false;
    }
    if (pos1 >= 0) fourier_tables(buf ^ 1, rec + b3n * C::RECS, pos1);
    // the real-space terms, from the last threads down (the first ones have
    // more of the Fourier tables)
    for (int t = THREADS - 1 - tid; t < nr; t += THREADS) {
      if (t < nrt1) real_term(r[0], ps.mog, (EIG && k_eig) ? pc + 8 : nullptr, kp, N, t, &rt);
      else if (COMP && t < nrt) real_term(r[1], ps.mog, nullptr, kp, N, t - nrt1, &rt, t);
      else real_term_zero(t, &rt);
    }
    if constexpr (LZ) {
      if (tid < 16) s_lzw[buf][tid] = p.lzw[((size_t)first + pos) * 16 + tid];
    }
    if (lead) publish(&s_pos[buf], pos3);
    async_copy_wait();
    sync_all();   // C1
    pos3 = s_pos[buf];
    if constexpr (LOSS) {
      if (lead) {
        write_chi2();   // the previous galaxy's
        if (!work) p.chi2[gal] = __int_as_float(0x7fc00000);   // NaN: a galaxy that is skipped
      }
    }

    // Lanczos and adding to the patch: the Fourier part of a galaxy with
    // real-space terms is parked in the workspace (this CTA's KL row pairs,
    // [2][KL][N]) until they are convolved
    const bool park = LZ && p.accumulate != 0 && nr > 0;
    float* const parked = reinterpret_cast<float*>(p.scratch256) + (size_t)blockIdx.x * 2 * KL * N;

    // ---- Step 7b: row pairs, inputs Z[k], k = j + m T; Step 8 ----
    if (work) {
      [[maybe_unused]] float* const mdl = (LOSS && p.model) ? p.model + off : nullptr;
      [[maybe_unused]] const float iv = LOSS ? p.ivar[gal] : 0.0f;
      [[maybe_unused]] float chi = 0.0f;
      float* const fourier = park ? parked : p.out + off;
#pragma unroll 1
      for (int rr = 0; rr < ROUNDS; ++rr) {
        const int pl = rr * GROUPS + f;
        const int pr = rank * KL + pl;   // rows pr and pr + N/2
        // element k = j + m T from column k (ZA, m < 8) or N - k (ZM)
        const uint32_t a = smem_u32(ZA + pr * SZ + j), b = smem_u32(ZM + pr * SZ + ((-j) & 15));
#pragma unroll
        for (int m = 0; m < 8; ++m) v[m] = cluster_ld2(cluster_map(a + 8 * block_slot(m), block_rank(m)));
        // N - k = 16 (16 - m) - j: block 15 - m, but 16 - m for j = 0 (N/2: rank 0's slot 0)
#pragma unroll
        for (int m = 8; m < 16; ++m) {
          const int b0 = (16 - m) & 7, b1 = 15 - m;
          v[m] = cluster_ld2(cluster_map(b + (j == 0 ? 8 * block_slot(b0) : 8 * block_slot(b1)),
                                         j == 0 ? block_rank(b0) : block_rank(b1)));
        }
        __syncwarp();   // the group's previous reads of its work row are done
        fft16<N, +1>(
            tw, v, [&](int k1) { return w + k1 * EX + j; }, [&](int q, int i) { return w + j * EX + i; }, [&] {
          // C2: the thread's last gathers have been issued before (the
          // exchange's writes depend on all of them)
          if (rr == ROUNDS - 1) cluster_arrive();
        });
        __syncwarp();
        float* const orow = reinterpret_cast<float*>(w);
        // x ^ cx ^ 4 [bit 5 of x], x = j + K: K's bit T and the 4 of bit 5
        // pick one of four bases, the rest of K is a compile-time offset
        float* const ob[4] = {orow + (j ^ cx), orow + (j ^ cx ^ 4), orow + (j ^ cx ^ T), orow + (j ^ cx ^ T ^ 4)};
#pragma unroll
        for (int k2 = 0; k2 < T; ++k2) {
          const int K = 16 * k2;
          float* const d = ob[((K >> 5) & 1) + 2 * (k2 & 1)] + (K & ~T);
          const float2 z = v[fft16_at<N>(0, k2)];
          d[0] = z.x;
          d[N] = z.y;
        }
        __syncwarp();   // the group's two rows are complete
        float* const dst = fourier + (size_t)(park ? pl : pr) * N;
#pragma unroll 1
        for (int i = 0; i < 2; ++i) {
          const int x0 = 8 * (j + T * i), p0 = x0 ^ cx ^ (((x0 >> 5) & 1) << 2);
          float2 o[8];
          {
            const float4 a0 = *reinterpret_cast<const float4*>(orow + p0), a1 = *reinterpret_cast<const float4*>(orow + (p0 ^ 4));
            const float4 b0 = *reinterpret_cast<const float4*>(orow + N + p0);
            const float4 b1 = *reinterpret_cast<const float4*>(orow + N + (p0 ^ 4));
            o[0] = make_float2(a0.x, b0.x); o[1] = make_float2(a0.y, b0.y); o[2] = make_float2(a0.z, b0.z);
            o[3] = make_float2(a0.w, b0.w); o[4] = make_float2(a1.x, b1.x); o[5] = make_float2(a1.y, b1.y);
            o[6] = make_float2(a1.z, b1.z); o[7] = make_float2(a1.w, b1.w);
          }
          if (!LZ && nrt > 0) real_space_rows(rt, nrt, (float)pr, (float)(pr + N / 2), (float)x0, o);
#pragma unroll
          for (int h = 0; h < 2; ++h) {
            float ov[8];
#pragma unroll
            for (int u = 0; u < 8; ++u) ov[u] = h ? o[u].y : o[u].x;
            if constexpr (LOSS)
              chi += loss_store8(dat, p.out + off, mdl, (int64_t)(pr + h * (N / 2)) * N + x0, ov, 2.0f * iv);
            else store8(dst + h * (park ? KL : N / 2) * N + x0, ov, p.accumulate != 0 && !park);
          }
        }
        __syncwarp();   // the group's reads of its work row are done
      }
      pending = true;
      if constexpr (LOSS) {
        for (int o2 = 16; o2 > 0; o2 >>= 1) chi += __shfl_xor_sync(0xffffffffu, chi, o2);
        if ((tid & 31) == 0) {
          float* slot = &s_chi[LOSS ? buf : 0][rank * WARPS + (tid >> 5)];
          cluster_st(cluster_map(smem_u32(slot), 0), chi);
        }
        if (lead) {
          chi_gal = gal;
          chi_iv = iv;
          chi_buf = buf;
        }
      }
    }
    if constexpr (LZ) {
      if (nr > 0) {   // uniform over the cluster
        // ---- the real-space part: the terms at the integer offset on the
        // group's rows, convolved along x there, kept where Z was, then along
        // y over the rows of every CTA, added to the stored Fourier part ----
        cluster_wait();   // every CTA has gathered its rows of Z
        float* const RR = reinterpret_cast<float*>(ZA);   // [row pair][2][N]
        const float* const wl = s_lzw[LZ ? buf : 0];
#pragma unroll 1
        for (int rr = 0; rr < ROUNDS; ++rr) {
          const int pl = rr * GROUPS + f;
          float* const rows = RR + pl * 2 * N;
#pragma unroll 1
          for (int i = 0; i < 2; ++i) {
            const int x0 = 8 * (j + T * i);
            float2 X[8];
#pragma unroll
            for (int u = 0; u < 8; ++u) X[u] = make_float2(0.0f, 0.0f);
            real_space_rows(rt, nrt, (float)(rank * KL + pl), (float)(rank * KL + pl + N / 2), (float)x0, X);
            float4* const d0 = reinterpret_cast<float4*>(rows + x0);
            float4* const d1 = reinterpret_cast<float4*>(rows + N + x0);
            d0[0] = make_float4(X[0].x, X[1].x, X[2].x, X[3].x);
            d0[1] = make_float4(X[4].x, X[5].x, X[6].x, X[7].x);
            d1[0] = make_float4(X[0].y, X[1].y, X[2].y, X[3].y);
            d1[1] = make_float4(X[4].y, X[5].y, X[6].y, X[7].y);
          }
          __syncwarp();
#pragma unroll 1
          for (int h = 0; h < 2; ++h) {
            float* const row = rows + h * N;
            float X[2][8];
            // along x: J(x) = sum_a w_a R(x - a) over the window x0 - 3 .. x0 + 10
#pragma unroll
            for (int i = 0; i < 2; ++i) {
              const int x0 = 8 * (j + T * i);
              const float4 c0 = *reinterpret_cast<const float4*>(row + x0);
              const float4 c1 = *reinterpret_cast<const float4*>(row + x0 + 4);
              float win[14];
              win[3] = c0.x; win[4] = c0.y; win[5] = c0.z; win[6] = c0.w;
              win[7] = c1.x; win[8] = c1.y; win[9] = c1.z; win[10] = c1.w;
#pragma unroll
              for (int a = 0; a < 3; ++a) {
                win[a] = row[(x0 - 3 + a) & (N - 1)];
                win[11 + a] = row[(x0 + 8 + a) & (N - 1)];
              }
#pragma unroll
              for (int u = 0; u < 8; ++u) {
                float acc = 0.0f;
#pragma unroll
                for (int a = 0; a < 7; ++a) acc = fmaf(wl[a], win[3 + u - (a - 3)], acc);
                X[i][u] = acc;
              }
            }
            __syncwarp();
#pragma unroll
            for (int i = 0; i < 2; ++i) {
              const int x0 = 8 * (j + T * i);
              *reinterpret_cast<float4*>(row + x0) = make_float4(X[i][0], X[i][1], X[i][2], X[i][3]);
              *reinterpret_cast<float4*>(row + x0 + 4) = make_float4(X[i][4], X[i][5], X[i][6], X[i][7]);
            }
          }
        }
        sync_all();   // every row has been convolved along x
        // along y: J(y) = sum_b w_b R(y - b), b = -3 .. 3
        const uint32_t rbase = smem_u32(RR);
#pragma unroll 1
        for (int rr = 0; rr < 2 * ROUNDS; ++rr) {
          const int pl = (rr >> 1) * GROUPS + f;
          const int y = rank * KL + pl + (rr & 1) * (N / 2);
          float* const dst = p.out + off + (size_t)y * N;
          const float* const src = park ? parked + (size_t)(pl + (rr & 1) * KL) * N : dst;
          float F[2][8];
#pragma unroll
          for (int i = 0; i < 2; ++i)
#pragma unroll
            for (int u = 0; u < 8; ++u) F[i][u] = 0.0f;
#pragma unroll 1
          for (int b = -3; b <= 3; ++b) {
            const int row = (y - b) & (N - 1), rp = row & (N / 2 - 1);
            const float wb = wl[8 + b + 3];
            const uint32_t a = cluster_map(rbase + 4 * ((rp % KL) * 2 * N + (row >= N / 2 ? N : 0)), rp / KL);
#pragma unroll
            for (int i = 0; i < 2; ++i) {
              const float4 u0 = cluster_ld4(a + 32 * (j + T * i)), u1 = cluster_ld4(a + 32 * (j + T * i) + 16);
              const float t[8] = {u0.x, u0.y, u0.z, u0.w, u1.x, u1.y, u1.z, u1.w};
#pragma unroll
              for (int u = 0; u < 8; ++u) F[i][u] = fmaf(wb, t[u], F[i][u]);
            }
          }
          // added to the Fourier part at the end, as in lanczos_real_strips: the
          // two kernels of this side round alike
#pragma unroll
          for (int i = 0; i < 2; ++i) {
            const float4* d = reinterpret_cast<const float4*>(src + 8 * (j + T * i));
            const float4 a = d[0], b = d[1];   // written by this thread
            const float o[8] = {a.x + F[i][0], a.y + F[i][1], a.z + F[i][2], a.w + F[i][3],
                                b.x + F[i][4], b.y + F[i][5], b.z + F[i][6], b.w + F[i][7]};
            store8(dst + 8 * (j + T * i), o, park);
          }
        }
        cluster_arrive();   // C2 again: the gathers of these rows are done
      }
    }
    pos = pos1;
    pos1 = pos2;
    pos2 = pos3;
    b3 = b3n;
  }
  if (pending) cluster_wait();   // no CTA ends while another gathers from it
  if constexpr (LOSS) {
    sync_all();   // the last galaxy's residuals are in
    if (lead) write_chi2();
  }
}

}  // namespace

template <bool LZ, bool EIG, bool LOSS = false, bool COMP = false>
static cudaError_t launch_fwd256c(const RenderParams& p, int num_sms, cudaStream_t s) {
  using C = CfgC<COMP>;
  auto fn = render_fwd256c_kernel<LZ, EIG, LOSS, COMP>;
  const int occ = kernel_occupancy(reinterpret_cast<const void*>(fn), THREADS, C::SMEM);
  if (occ < 0) return cudaErrorInvalidConfiguration;
  const int clusters = persistent_grid(p, occ < CTAS_PER_SM ? occ : CTAS_PER_SM, num_sms / CL);
  // (the parked Fourier parts of the Lanczos variant, KL row pairs per CTA, fit
  // the scratch's CTAS_PER_SM slices of a whole patch per SM)
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3((unsigned)(clusters * CL));
  cfg.blockDim = dim3(THREADS);
  cfg.dynamicSmemBytes = C::SMEM;
  cfg.stream = s;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = CL;
  at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, fn, p);
}

cudaError_t launch_render_fwd256_small(const RenderParams& p, int num_sms, cudaStream_t s) {
  if (p.records2)
    return p.lanczos ? launch_fwd256c<true, false, false, true>(p, num_sms, s)
                     : launch_fwd256c<false, false, false, true>(p, num_sms, s);
  if (p.loss)
    return p.eigen ? launch_fwd256c<false, true, true>(p, num_sms, s) : launch_fwd256c<false, false, true>(p, num_sms, s);
  if (p.eigen)
    return p.lanczos ? launch_fwd256c<true, true>(p, num_sms, s) : launch_fwd256c<false, true>(p, num_sms, s);
  return p.lanczos ? launch_fwd256c<true, false>(p, num_sms, s) : launch_fwd256c<false, false>(p, num_sms, s);
}

}  // namespace mog
