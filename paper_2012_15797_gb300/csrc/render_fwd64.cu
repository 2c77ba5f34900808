// Fused forward render of 64 x 64 patches (Section 2, Steps 3-8), 16 values per
// thread (fft16.cuh): a 128-thread CTA per galaxy, 4 threads per transform, the
// schedule of render_fwd128.cu with one column and one row pair per thread
// group.  Everything is done in place in the N/2 rows of Z (17 KB), row p the
// input of the transform of row pair (p, p + N/2).
//
// Two CTA barriers per galaxy: between the columns and the rows, and before the
// next galaxy's columns write (after their evaluation).  The PSF spectrum is kept
// in shared memory; when the next galaxy has another, it is on its way during the
// rows of this one (an eigen-PSF's is formed there for each galaxy).  The
// twiddles are read from shared memory before each transform: as 30 registers of
// every thread they left room for four CTAs per SM, without them for five (89
// registers, no spills).
//
// Issue slots, shared memory and latency at 20 warps per SM bound it (issue 65%,
// l1tex 70%).  Against 8 values per
// thread (256 threads, four CTAs per SM, three barriers and twice the table and
// component reads): 7.9k instead of 8.7k warp instructions and 1.9k instead of
// 2.2k shared-memory wavefronts per galaxy; 100k galaxies 0.976 -> 0.930 ms, the
// call 1.039 -> 0.996 (1.068 with the PSF spectrum read through L1, 1.018 with it in shared
// memory at four CTAs, 1.065 at five with the twiddles in registers, spilled),
// the fit step of 50k 1.671 -> 1.638, 40k of an eigen-PSF 0.695 -> 0.658; with the
// Lanczos shift (four CTAs) 100k 1.321 -> 1.288 (1.333 with the phases along omega
// formed twice, for the table and for the nu = 1/2 column), 300 galaxies 36 -> 31 us.
#include "fwd16.cuh"

namespace mog {

namespace {

constexpr int N = 64;
constexpr int T = fft16_threads<N>();      // 4 threads per transform
constexpr int NP = N / 2;                  // columns, row pairs
constexpr int THREADS = NP * T;            // 128
constexpr int WARPS = THREADS / 32;
constexpr int LS = psf_lstride(N);
constexpr int B = bucket_of(N);
constexpr int HALF = N / 2 + 2;            // omega = 0 .. 1/2 (padded)
// Row stride of Z and of the staged PSF spectrum in float2, 4 modulo 16: a
// half-warp (one wavefront of 8-byte accesses) is four groups of T threads, and
// the 4 rows x 4 columns that it touches take 16 different bank pairs.
constexpr int RS = N + 16 / T;

struct Smem64 {
  float2 z[NP * RS];
  float2 psf[NP * RS];             // columns 0 .. N/2 - 1 of the PSF spectrum in use
  // per galaxy, two buffers: phases along omega and nu, the nu = 1/2 column,
  // Fourier components; records: three
  float2 py[2 * HALF], px[2 * NP], hn[2 * HALF];
  float4 fc[2 * KMAX];
  GalaxyRecord rec[3];
  RealTerms rt;
  float4 tw[8 * T];                // twiddles 2 i, 2 i + 1 of thread j at [i T + j]
};
// The Lanczos shift adds the real-space part's rows.
template <bool LZ>
struct Cfg64 {
  static constexpr int CTAS_PER_SM = LZ ? 4 : 5;
  static constexpr size_t SMEM = sizeof(Smem64) + (LZ ? sizeof(float) * N * N : 0);
  static_assert(CTAS_PER_SM * (SMEM + 320 + 1024) <= 228 * 1024, "they share an SM's shared memory");
};
static_assert(sizeof(Smem64) % 16 == 0, "the rows start on a 16-byte boundary");

// Pixel x of an output row staged in row p of Z is kept at x ^ 4 [bit 0 of p xor
// bit 2 of p]: the rows p and p + 4 that a warp writes and the rows p and p + 1
// that a quarter-warp reads in 16-byte pieces then take different banks.
__device__ __forceinline__ int staged(int p) { return ((p ^ (p >> 2)) & 1) << 2; }

// LZ: the Lanczos sub-pixel shift (records carry the integer offset and the
// fraction): the convolution of the Fourier part is folded into the phase
// tables, the real-space part is convolved and added where the Fourier
// part is staged.  EIG: some PSF of the context is an eigen-PSF.
// LOSS: the loss mode of mog_render_chi2.
template <bool LZ, bool EIG, bool LOSS>
__global__ void __launch_bounds__(THREADS, Cfg64<LZ>::CTAS_PER_SM) render_fwd64_kernel(RenderParams p) {
  static_assert(!(LZ && LOSS), "the loss mode renders with the phase shift");
  constexpr float INV_N = 1.0f / N;
  extern __shared__ __align__(128) unsigned char smem[];
  Smem64& S = *reinterpret_cast<Smem64*>(smem);
  float2* const Z = S.z;
  GalaxyRecord* const rec = S.rec;
  __shared__ int s_first[3], s_pos[2];
  __shared__ float s_lzw[LZ ? 2 : 1][16];   // per buffer: Lanczos weights along x [0, 7) and y [8, 15)
  __shared__ float s_chi[LOSS ? 2 : 1][WARPS];   // each warp's sum of squared residuals

  const int tid = threadIdx.x;
  const int f = tid / T, j = tid % T;
  for (int i = tid; i < 8 * T; i += THREADS) {
    float4 w;
    const int jj = i % T, k = 2 * (i / T);
    sincospif(2.0f * (float)(jj * k) * INV_N, &w.y, &w.x);
    sincospif(2.0f * (float)(jj * (k + 1)) * INV_N, &w.w, &w.z);
    S.tw[i] = w;
  }
  auto load_tw = [&](float2 (&tw)[15]) {
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const float4 w = S.tw[i * T + j];
      if (i > 0) tw[2 * i - 1] = make_float2(w.x, w.y);
      tw[2 * i] = make_float2(w.z, w.w);
    }
  };
  const int count = p.bucket_count[B];
  const int first = p.bucket_start[B];          // planned position of this bucket's first galaxy
  const unsigned char* records = p.records + (size_t)first * RECORD_BYTES;

  // The work queue is taken by thread 0, p.chunk positions at a time with the
  // next chunk requested one chunk ahead; a position is published three
  // galaxies ahead.
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
  // the record of planned position pos into buffer b (16-byte pieces, one per
  // thread)
  auto load_record = [&](int b, int pos) {
    if (tid < (int)sizeof(GalaxyRecord) / 16)
      async_copy16(reinterpret_cast<float4*>(rec + b) + tid,
                   reinterpret_cast<const float4*>(records + (size_t)pos * RECORD_BYTES) + tid);
  };
  // LOSS, thread 0, once every warp has added its residuals of chi_gal
  long long chi_gal = -1;
  float chi_iv = 0.0f;
  int chi_buf = 0;
  auto write_chi2 = [&]() {
    if (chi_gal >= 0) {
      float t = 0.0f;
      for (int i = 0; i < WARPS; ++i) t += s_chi[chi_buf][i];
      p.chi2[chi_gal] = chi_iv * t;
      chi_gal = -1;
    }
  };

  // Tables of a galaxy.  Phases and the nu = 1/2 column are kept for omega =
  // 0 .. 1/2: at -omega they are the complex conjugates.  hn: the Hermitian part
  // of the nu = 1/2 column, the mean of its value at omega and the conjugate at
  // -omega.
  auto shift_phase = [](float g, float fr, const float* lzw) {
    float2 ph;
    sincospif(-2.0f * g * fr, &ph.y, &ph.x);
    if constexpr (LZ) {
      float wv[7];
      load_weights(lzw, 0, wv);
      ph = cmul(ph, lanczos_response(wv, fr));
    }
    return ph;
  };
  auto fourier_tables = [&](int b, const GalaxyRecord& r, int pos) {
    if (!r.ok) return;
    const DevPsf& ps = p.psfs[r.psf];
    const float2* const spec = ps.spec[B];
    const int k_eig = EIG ? ps.k_eig : 0;
    const float* pc = p.pcoef + ((size_t)first + pos) * PCOEF;
    const float* lzw = LZ ? p.lzw + ((size_t)first + pos) * 16 : nullptr;
    const float gx = r.x, gy = r.y;
    constexpr int NH = N / 2 + 1;
    constexpr int t1 = NH, t2 = t1 + NP;
    for (int i = tid; i < t2 + r.nf; i += THREADS) {
      if (i < t1) {
        const int l = i;
        const float om = (float)l * INV_N;
        float2 val[2];
        const float2 phx = shift_phase(gx, 0.5f, lzw), phy = shift_phase(gy, om, LZ ? lzw + 8 : nullptr);
        S.py[b * HALF + l] = phy;
#pragma unroll
        for (int h = 0; h < 2; ++h) {   // at omega and -omega; N/2 is one bin, omega = -1/2
          const bool neg = h || l == N / 2;
          const float o = neg ? -om : om;
          const float q = fmaf(o, fmaf(r.s22, o, r.s12), 0.25f * r.s11);
          float acc = 0.0f;
          for (int c = 0; c < r.nf; ++c) acc = fmaf(r.famp[c], ex2(r.fcoef[c] * q), acc);
          const int e = (N / 2) * LS + (h ? (N - l) & (N - 1) : l);
          const float2 pn = (EIG && k_eig) ? eigen_bin(spec, psf_spec_elems(N), k_eig, pc, e) : __ldg(spec + e);
          val[h] = cscale(cmul(pn, cmul(phx, neg ? conjf2(phy) : phy)), acc);
        }
        S.hn[b * HALF + l] = make_float2(0.5f * (val[0].x + val[1].x), 0.5f * (val[0].y - val[1].y));
      } else if (i < t2) {
        S.px[b * NP + i - t1] = shift_phase(gx, (float)(i - t1) * INV_N, lzw);
      } else {
        const int c = i - t2;
        S.fc[b * KMAX + c] = make_float4(r.famp[c], r.famp[c], r.fcoef[c], r.fcoef[c]);
      }
    }
  };

  if (tid == 0) {
    q_ahead = atomicAdd(&p.queue[B], p.chunk);
    for (int i = 0; i < 3; ++i) s_first[i] = next_position();
  }
  __syncthreads();
  int pos = s_first[0], pos1 = s_first[1], pos2 = s_first[2];
  if (pos >= 0) load_record(0, pos);
  if (pos1 >= 0) load_record(1, pos1);
  async_copy_wait();
  __syncthreads();
  if (pos >= 0) fourier_tables(0, rec[0], pos);
  // The PSF spectrum of a galaxy, on its way into shared memory unless it is
  // there; complete for a thread's own pieces after async_copy_wait.  An
  // eigen-PSF's is formed for each galaxy.
  int staged_psf = -1;
  auto stage_psf = [&](const GalaxyRecord& r, int pos) {
    if (!r.ok || r.psf == staged_psf) return false;
    const DevPsf& ps = p.psfs[r.psf];
    const float2* const spec = ps.spec[B];
    if (EIG && ps.k_eig) {
      staged_psf = -1;
      const float* pc = p.pcoef + ((size_t)first + pos) * PCOEF;
      constexpr int COLS = THREADS / N, M = 8;   // columns at a time
      const int c0 = tid / N, l = tid % N;
#pragma unroll 1
      for (int c = c0; c < NP; c += M * COLS) {
        float2 s[M];
        eigen_bins(spec + c * LS + l, psf_spec_elems(N), ps.k_eig, pc, [](int i) { return i * COLS * LS; }, s);
#pragma unroll
        for (int i = 0; i < M; ++i) S.psf[(c + i * COLS) * RS + l] = s[i];
      }
      return true;
    }
    staged_psf = r.psf;
    for (int i = tid; i < NP * (N / 2); i += THREADS) {
      const int c = i / (N / 2), e = 2 * (i % (N / 2));
      async_copy16(S.psf + c * RS + e, spec + c * LS + e);
    }
    return true;
  };
  bool staging = pos >= 0 && stage_psf(rec[0], pos);
  __syncthreads();

  // Who waits for whom.  Per galaxy i the CTA meets before its columns write
  // (C2(i - 1): every thread has left the rows of i - 1) and between its
  // columns and its rows (C1(i)).  Before C1(i): the columns of i (reading its
  // Fourier tables and record), the Fourier tables of i + 1 (buffer (i + 1) & 1,
  // last read before C1(i - 1); from the record of i + 1, loaded before
  // C1(i - 1)), after C2(i - 1) the real-space terms of i, and the record of
  // i + 2 (the buffer of i - 1, last read before C1(i - 1)).  The rows use no
  // record: what they need of it is in registers.
  int b3 = 0;
  for (int buf = 0; pos >= 0; buf ^= 1) {
    const GalaxyRecord& r = rec[b3];
    const int b3n = b3 == 2 ? 0 : b3 + 1;
    const bool work = r.ok != 0;   // uniform
    const DevPsf& ps = p.psfs[work ? r.psf : 0];
    const int k_eig = EIG ? ps.k_eig : 0;
    const float* pc = p.pcoef + ((size_t)first + pos) * PCOEF;
    const int kp = ps.k, nrt = work ? r.nrc * kp : 0;
    const int64_t off = r.off;
    [[maybe_unused]] const int64_t gal = r.gal;
    if (staging) {   // uniform
      async_copy_wait();
      __syncthreads();
      staging = false;
    }
    if (pos2 >= 0) load_record(b3n == 2 ? 0 : b3n + 1, pos2);
    int pos3 = -1;
    if (tid == 0) pos3 = next_position();
    [[maybe_unused]] const float* const dat = (LOSS && work) ? (p.dptr ? p.dptr[gal] : p.data + off) : nullptr;
    if constexpr (LOSS) {
      // the data patch's lines, on their way to L2
      if (work)
        for (int i = tid; i < N * N / 32; i += THREADS) prefetch_l2(dat + 32 * i);
    }

    // ---- Steps 5-6 on the bins l = j + m T of the group's column f, Step 7a ----
    float2 v[16];
    if (work) {
      const float2* const py = S.py + buf * HALF;
      const float2 pxk = S.px[buf * NP + f];
      float2 s[8];
#pragma unroll
      for (int k = 0; k < 8; ++k) s[k] = make_float2(0.0f, 0.0f);
      mixture16(S.fc + buf * KMAX, r.nf, r.s11, 2.0f * r.s12, r.s22, (float)f * INV_N, (float)j * INV_N, s);
#pragma unroll
      for (int m = 0; m < 16; ++m) {
        const int l = j + m * T;
        const float2 e = m < 8 ? cmul(pxk, py[l]) : cmulc(pxk, py[N - l]);
        v[m] = cscale(cmul(S.psf[f * RS + l], e), (m & 1) ? s[m >> 1].y : s[m >> 1].x);
      }
      if (f == 0) {
        // Pack the Hermitian parts of the nu = 0 and nu = 1/2 columns as
        // re + i im.  The nu = 0 column is Hermitian in omega by construction
        // (its self-conjugate bin l = N/2 keeps its real part).
        const float2* const hn = S.hn + buf * HALF;
#pragma unroll
        for (int m = 0; m < 16; ++m) {
          const int l = j + m * T;
          const float2 dc = (l == N / 2) ? make_float2(v[m].x, 0.0f) : v[m];
          const float2 h = m < 8 ? hn[l] : conjf2(hn[N - l]);
          v[m] = make_float2(dc.x - h.y, dc.y + h.x);
        }
      }
      __syncthreads();   // C2 of the previous galaxy
      // Exchange element (k1, j): row ((k1 mod 8) T + j ^ (k1 mod T)) of the
      // column's place f (k1 < 8) or N - f.
      float2* const zk = Z + f;
      float2* const zm = Z + (f ? N - f : N / 2);
      float2 tw[15];
      load_tw(tw);
      fft16<N, +1>(
          tw, v, [&](int k1) { return ((k1 & 8) ? zm : zk) + ((k1 & 7) * T + (j ^ (k1 & (T - 1)))) * RS; },
          [&](int q, int i) { return (((T * q) & 8) ? zm : zk) + ((j + ((T * q) & 7)) * T + (j ^ i)) * RS; });
      // rows n = j + T q + 16 k2 of the column: pairs (p, p + N/2) are k2, k2 + T/2
#pragma unroll
      for (int q = 0; q < 16 / T; ++q)
#pragma unroll
        for (int k2 = 0; k2 < T / 2; ++k2) {
          const float2 A = v[fft16_at<N>(q, k2)], Bv = v[fft16_at<N>(q, k2 + T / 2)];
          const int o = (j + T * q + 16 * k2) * RS;
          zk[o] = f ? make_float2(A.x - Bv.y, A.y + Bv.x) : make_float2(A.x, Bv.x);
          zm[o] = f ? make_float2(A.x + Bv.y, Bv.x - A.y) : make_float2(A.y, Bv.y);
        }
      // the real-space terms, from the last threads down (the first ones have
      // more of the Fourier tables)
      const int nr2 = real_terms_padded(nrt);
      for (int t = THREADS - 1 - tid; t < nr2; t += THREADS) {
        if (t < nrt) real_term(r, ps.mog, (EIG && k_eig) ? pc + 8 : nullptr, kp, N, t, &S.rt);
        else real_term_zero(t, &S.rt);
      }
      if constexpr (LZ) {
        if (tid < 16) s_lzw[buf][tid] = p.lzw[((size_t)first + pos) * 16 + tid];
      }
    } else {
      __syncthreads();   // C2
    }
    if (pos1 >= 0) fourier_tables(buf ^ 1, rec[b3n], pos1);
    if (tid == 0) s_pos[buf] = pos3;
    async_copy_wait();
    __syncthreads();   // C1
    pos3 = s_pos[buf];
    if (pos1 >= 0) staging = stage_psf(rec[b3n], pos1);   // galaxies are planned by PSF: seldom
    if constexpr (LOSS) {
      if (tid == 0) {
        write_chi2();   // the previous galaxy's
        if (!work) p.chi2[gal] = __int_as_float(0x7fc00000);   // NaN: a galaxy that is skipped
      }
    }

    // ---- Step 7b: row pair f, inputs Z[k], k = j + m T; Step 8 ----
    if (work) {
      [[maybe_unused]] float* const mdl = (LOSS && p.model) ? p.model + off : nullptr;
      [[maybe_unused]] const float iv = LOSS ? p.ivar[gal] : 0.0f;
      [[maybe_unused]] float chi = 0.0f;
      float2* const zr = Z + f * RS;
#pragma unroll
      for (int m = 0; m < 16; ++m) v[m] = zr[j + m * T];
      __syncwarp();
      float2 tw[15];
      load_tw(tw);
      fft16<N, +1>(
          tw, v, [&](int k1) { return zr + k1 * T + (j ^ (k1 & (T - 1))); },
          [&](int q, int i) { return zr + (j + T * q) * T + (j ^ i); });
      // x = j + K, kept at x ^ sw: K ^ sw is K + sw or K - sw, so one of two
      // bases, K itself is a compile-time offset
      float* const orow = reinterpret_cast<float*>(zr);
      const int sw = staged(f);
      float* const ob[2] = {orow + j + sw, orow + j - sw};
#pragma unroll
      for (int q = 0; q < 16 / T; ++q)
#pragma unroll
        for (int k2 = 0; k2 < T; ++k2) {
          const int K = T * q + 16 * k2;
          float* const d = ob[(K >> 2) & 1] + K;
          const float2 z = v[fft16_at<N>(q, k2)];
          d[0] = z.x;
          d[N] = z.y;
        }
      if (!LZ || nrt == 0) {   // uniform; else stored below
        __syncwarp();   // the group's two rows are complete
        float* const dst = p.out + off + (size_t)f * N;
#pragma unroll 1
        for (int i = 0; i < 2; ++i) {
          const int x0 = 8 * (j + T * i), p0 = x0 ^ sw;
          float2 o[8];
          {
            const float4 a0 = *reinterpret_cast<const float4*>(orow + p0), a1 = *reinterpret_cast<const float4*>(orow + (p0 ^ 4));
            const float4 b0 = *reinterpret_cast<const float4*>(orow + N + p0);
            const float4 b1 = *reinterpret_cast<const float4*>(orow + N + (p0 ^ 4));
            o[0] = make_float2(a0.x, b0.x); o[1] = make_float2(a0.y, b0.y); o[2] = make_float2(a0.z, b0.z);
            o[3] = make_float2(a0.w, b0.w); o[4] = make_float2(a1.x, b1.x); o[5] = make_float2(a1.y, b1.y);
            o[6] = make_float2(a1.z, b1.z); o[7] = make_float2(a1.w, b1.w);
          }
          if (!LZ && nrt > 0) real_space_rows(S.rt, nrt, (float)f, (float)(f + N / 2), (float)x0, o);
#pragma unroll
          for (int h = 0; h < 2; ++h) {
            float ov[8];
#pragma unroll
            for (int u = 0; u < 8; ++u) ov[u] = h ? o[u].y : o[u].x;
            if constexpr (LOSS)
              chi += loss_store8(dat, p.out + off, mdl, (int64_t)(f + h * (N / 2)) * N + x0, ov, 2.0f * iv);
            else store8(dst + h * (N / 2) * N + x0, ov, p.accumulate != 0);
          }
        }
      }
      if constexpr (LOSS) {
        for (int o2 = 16; o2 > 0; o2 >>= 1) chi += __shfl_xor_sync(0xffffffffu, chi, o2);
        if ((tid & 31) == 0) s_chi[LOSS ? buf : 0][tid >> 5] = chi;
        if (tid == 0) {
          chi_gal = gal;
          chi_iv = iv;
          chi_buf = buf;
        }
      }
    }
    if constexpr (LZ) {
      if (nrt > 0) {   // uniform
        // the convolved real-space part, added to the Fourier part staged in Z
        // (all there after the first barrier inside)
        float* const dst = p.out + off;
        lanczos_real_strips<N, N, THREADS>(
            S.rt, nrt, s_lzw[LZ ? buf : 0], reinterpret_cast<float*>(smem + sizeof(Smem64)),
            [&](int y, int x0, const float(&acc)[8]) {
              const int pr = y & (NP - 1), p0 = x0 ^ staged(pr);
              const float* const row = reinterpret_cast<const float*>(Z + pr * RS) + (y >= NP ? N : 0);
              const float4 a = *reinterpret_cast<const float4*>(row + p0), c = *reinterpret_cast<const float4*>(row + (p0 ^ 4));
              const float ov[8] = {a.x + acc[0], a.y + acc[1], a.z + acc[2], a.w + acc[3],
                                   c.x + acc[4], c.y + acc[5], c.z + acc[6], c.w + acc[7]};
              store8(dst + (size_t)y * N + x0, ov, p.accumulate != 0);
            });
      }
    }
    pos = pos1;
    pos1 = pos2;
    pos2 = pos3;
    b3 = b3n;
  }
  if constexpr (LOSS) {
    __syncthreads();   // the last galaxy's residuals are in
    if (tid == 0) write_chi2();
  }
}

}  // namespace

template <bool LZ, bool EIG, bool LOSS = false>
static int fwd64_occupancy() {
  using C = Cfg64<LZ>;
  const int occ = kernel_occupancy(reinterpret_cast<const void*>(render_fwd64_kernel<LZ, EIG, LOSS>), THREADS, C::SMEM);
  return occ < 0 ? occ : (occ < C::CTAS_PER_SM ? occ : C::CTAS_PER_SM);
}

template <bool LZ, bool EIG, bool LOSS = false>
static cudaError_t launch_fwd64(const RenderParams& p, int num_sms, int ctas_per_sm, cudaStream_t s) {
  const int occ = fwd64_occupancy<LZ, EIG, LOSS>();
  if (occ < 0) return cudaErrorInvalidConfiguration;
  const int ctas = (ctas_per_sm > 0 && ctas_per_sm < occ) ? ctas_per_sm : occ;
  render_fwd64_kernel<LZ, EIG, LOSS><<<persistent_grid(p, ctas, num_sms), THREADS, Cfg64<LZ>::SMEM, s>>>(p);
  return cudaGetLastError();
}

cudaError_t launch_render_fwd64(const RenderParams& p, int num_sms, int ctas_per_sm, cudaStream_t s) {
  if (p.loss)
    return p.eigen ? launch_fwd64<false, true, true>(p, num_sms, ctas_per_sm, s)
                   : launch_fwd64<false, false, true>(p, num_sms, ctas_per_sm, s);
  if (p.eigen)
    return p.lanczos ? launch_fwd64<true, true>(p, num_sms, ctas_per_sm, s)
                     : launch_fwd64<false, true>(p, num_sms, ctas_per_sm, s);
  return p.lanczos ? launch_fwd64<true, false>(p, num_sms, ctas_per_sm, s)
                   : launch_fwd64<false, false>(p, num_sms, ctas_per_sm, s);
}

int render_fwd64_max_ctas() { return fwd64_occupancy<false, false>(); }

}  // namespace mog
