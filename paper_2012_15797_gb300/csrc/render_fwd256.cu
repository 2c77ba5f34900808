// Fused forward render for 256 x 256 patches (Section 2, Steps 3-8), 16 values
// per thread (fft16.cuh), two 256-thread CTAs per SM, one galaxy at a time per
// CTA, 16 threads per transform.
//
// The half spectrum (129 x 256 complex, 264 KB) does not fit in one CTA's
// shared memory, so the transform between the two FFT directions goes through
// the galaxy's own output patch, which stays L2-resident: the input of the
// row transform of row pair p (rows p and p + N/2; 256 complex, 2 KB)
// occupies exactly the bytes of those two output rows (elements below N/2 in
// row p, the rest in row p + N/2), which only that row transform overwrites.
//
//   columns   8 rounds of 16 columns.  First pass: 16 threads per column
//             evaluate its bins (Steps 5-6) and exchange through shared memory
//             (two buffers, one CTA barrier per round).  Second pass: 16
//             columns side by side per half-warp, so that the row-pair inputs,
//             formed in the thread, are stored as 128-byte segments directly
//   rows      8 rounds of 16 row pairs, each half-warp on its own: load the
//             row pair's input, transform, add the real-space terms, store
//             the two pixel rows over the input
// The PSF spectrum (272 KB) is read from global memory (L2-resident).
//
// What bounds it: issue slots and latency at the 16 warps per SM that 128
// registers a thread leave (issue 54%, shared memory 50%, FMA pipe 44%; DRAM
// below 20%).  Against 8 values per thread (radix 8 x 8 x 4, two exchanges per
// transform, the row-pair inputs staged through shared memory with two CTA
// barriers per round, 512 threads at 64 registers): 129k warp instructions and
// 18k shared-memory wavefronts per galaxy instead of 199k and 43k; the 10.6k
// 256 x 256 galaxies of the 200k mixed workload 2.47 -> 2.00 ms (with the loss
// 2.83 -> 2.68, composites 2.94 -> 2.65 ms; a call with the Lanczos shift on 10.6k
// galaxies of one profile 2.97 -> 2.31).
//
// Lanczos variant (LZ): the Fourier part is shifted through the phase tables
// (the Lanczos transfer function H(nu) H(omega)); a galaxy with real-space
// terms then gets its real-space part convolved and added in strips of
// 64 rows: the 70 rows each strip needs are evaluated and convolved along x
// (one warp per row, neighbours by shuffle) into shared memory that the
// transforms no longer use, then convolved along y and added to the patch.
#include "fwd16.cuh"

namespace mog {

namespace {

constexpr int N = 256;
constexpr int T = fft16_threads<N>();      // 16
constexpr int THREADS = 256;
constexpr int GROUPS = THREADS / T;        // 16 transforms at a time
constexpr int WARPS = THREADS / 32;
constexpr int ROUNDS = (N / 2) / GROUPS;   // 8
constexpr int CTAS_PER_SM = 2;
constexpr int LS = psf_lstride(N);
constexpr int PSF_ELEMS = psf_spec_elems(N);
constexpr int B = bucket_of(N);
constexpr int HALF = N / 2 + 2;            // omega = 0 .. 1/2 (padded)
constexpr int STRIP = 64;                  // Lanczos: output rows per strip
constexpr int CHI_SUMS = ROUNDS / 2 * WARPS;

// float2 offset of element c of row pair p's transform input in the patch
__device__ __forceinline__ int zpos(int p, int c) { return (c < N / 2 ? p : p + N / 2) * (N / 2) + (c & (N / 2 - 1)); }

// Exchange row of one transform: element (k1, i) at 17 k1 + i, conflict free
// both ways for the 16 threads of a transform.  The columns' rows are 273
// float2 apart (odd: the second pass reads 16 columns side by side), the
// rows' 272 (16-byte pieces).
constexpr int EX = T + 1;
constexpr int CS = 16 * EX + 1, RSTR = 16 * EX;

template <bool COMP>
struct Cfg256 {
  using RT = RealTermsN<COMP ? 2 * RMAX : RMAX>;
  static constexpr int RECS = COMP ? 2 : 1;   // records per galaxy
  static constexpr size_t off_w = 0;          // two buffers of 16 exchange rows; Lanczos strips
  static constexpr size_t W_BYTES = 2 * sizeof(float2) * GROUPS * CS > sizeof(float) * (STRIP + 6) * N
                                        ? 2 * sizeof(float2) * GROUPS * CS : sizeof(float) * (STRIP + 6) * N;
  // per galaxy, two buffers: phases along omega and nu, the nu = 1/2 column,
  // Fourier components; records: three
  static constexpr size_t off_py = off_w + W_BYTES;
  static constexpr size_t off_px = off_py + 2 * sizeof(float2) * HALF;
  static constexpr size_t off_hn = off_px + 2 * sizeof(float2) * (N / 2);
  static constexpr size_t off_fc = (off_hn + 2 * sizeof(float2) * HALF + 15) & ~size_t(15);
  static constexpr size_t off_rec = off_fc + 2 * sizeof(float4) * RECS * KMAX;
  static constexpr size_t off_rt = off_rec + 3 * RECS * sizeof(GalaxyRecord);
  static constexpr size_t SMEM = off_rt + sizeof(RT);
  static_assert(STRIP % 2 == 0, "rows in pairs");
  static_assert(CTAS_PER_SM * (SMEM + 512 + 1024) <= 228 * 1024, "two CTAs share an SM's shared memory");
};

// LZ: the Lanczos sub-pixel shift (records carry the integer offset and the
// fraction): the convolution of the Fourier part is folded into the phase
// tables, the real-space part is convolved along x, then along y, in strips.
// EIG: some PSF of the context is an eigen-PSF.  LOSS: the loss mode of mog_render_chi2.  COMP: composites of two profiles
// (p.records2).
template <bool LZ, bool EIG, bool LOSS, bool COMP>
__global__ void __launch_bounds__(THREADS, CTAS_PER_SM) render_fwd256_kernel(RenderParams p) {
  using C = Cfg256<COMP>;
  using RT = typename C::RT;
  static_assert(!(LZ && LOSS), "the loss mode renders with the phase shift");
  static_assert(!(COMP && (EIG || LOSS)), "composites: constant PSFs, plain render");
  constexpr int NP = N / 2;
  constexpr float INV_N = 1.0f / N;
  extern __shared__ __align__(128) unsigned char smem[];
  float2* W = reinterpret_cast<float2*>(smem + C::off_w);
  float2* pys = reinterpret_cast<float2*>(smem + C::off_py);   // [buffer][omega N = 0 .. N/2]
  float2* pxs = reinterpret_cast<float2*>(smem + C::off_px);   // [buffer][NP]
  float2* hns = reinterpret_cast<float2*>(smem + C::off_hn);   // [buffer][omega N = 0 .. N/2]
  float4* fcs = reinterpret_cast<float4*>(smem + C::off_fc);   // [buffer][RECS * KMAX]
  GalaxyRecord* rec = reinterpret_cast<GalaxyRecord*>(smem + C::off_rec);   // [3][RECS]
  RT& rt = *reinterpret_cast<RT*>(smem + C::off_rt);
  __shared__ int s_first[3], s_pos[2];
  __shared__ float s_lzw[LZ ? 2 : 1][16];   // per buffer: Lanczos weights along x [0, 7) and y [8, 15)
  __shared__ float s_chi[LOSS ? 2 : 1][LOSS ? CHI_SUMS : 1];   // sums of squared residuals: [rounds 2 i, 2 i + 1][warp]

  const int tid = threadIdx.x;
  const int f = tid / T, j = tid % T;
  float2 tw[15];
  fft16_twiddles<N>(j, tw);
  const int cx = (f & 1) * T;   // staged output rows, see below
  const int count = p.bucket_count[B];
  if (count < p.bucket_min || count > p.bucket_max) return;   // the other kernel's (launch_by_count)
  const int first = p.bucket_start[B];          // planned position of this bucket's first galaxy
  const unsigned char* records = p.records + (size_t)first * RECORD_BYTES;
  [[maybe_unused]] const unsigned char* records2 = COMP ? p.records2 + (size_t)first * RECORD_BYTES : nullptr;

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
  // the record(s) of planned position pos into buffer b (16-byte pieces, one
  // per thread)
  auto load_records = [&](int b, int pos) {
    constexpr int PIECES = sizeof(GalaxyRecord) / 16;
    float4* const d = reinterpret_cast<float4*>(&rec[b * C::RECS]) + tid;
    if (tid < PIECES) async_copy16(d, reinterpret_cast<const float4*>(records + (size_t)pos * RECORD_BYTES) + tid);
    else if (COMP && tid < 2 * PIECES)
      async_copy16(d, reinterpret_cast<const float4*>(records2 + (size_t)pos * RECORD_BYTES) + tid - PIECES);
  };
  // LOSS, thread 0, once every warp has added its residuals of chi_gal
  long long chi_gal = -1;
  float chi_iv = 0.0f;
  int chi_buf = 0;
  auto write_chi2 = [&]() {
    if (chi_gal >= 0) {
      float t = 0.0f;
      for (int i = 0; i < CHI_SUMS; ++i) t += s_chi[chi_buf][i];
      p.chi2[chi_gal] = chi_iv * t;
      chi_gal = -1;
    }
  };

  // Tables of a galaxy.  Phases and the nu = 1/2 column are kept for omega =
  // 0 .. 1/2: at -omega they are the complex conjugates (also the Lanczos
  // responses, whose weights are real).  hn: the Hermitian part of the nu =
  // 1/2 column, the mean of its value at omega and the conjugate at -omega.
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
    constexpr int t1 = NH, t2 = t1 + NH, t3 = t2 + NP;
    for (int i = tid; i < t3 + nfa; i += THREADS) {
      if (i < t1) {
        const int l = i;
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
      } else if (i < t2) {
        pys[b * HALF + i - t1] = shift_phase(gy, (float)(i - t1) * INV_N, LZ ? lzw + 8 : nullptr);
      } else if (i < t3) {
        pxs[b * NP + i - t2] = shift_phase(gx, (float)(i - t2) * INV_N, lzw);
      } else {
        const int c = i - t3;
        const GalaxyRecord& rr = r[(COMP && c >= nf1) ? 1 : 0];
        const int cc = c - (COMP && c >= nf1 ? nf1 : 0);
        fcs[b * C::RECS * KMAX + c] = make_float4(rr.famp[cc], rr.famp[cc], rr.fcoef[cc], rr.fcoef[cc]);
      }
    }
  };

  if (tid == 0) {
    q_ahead = atomicAdd(&p.queue[B], p.chunk);
    for (int i = 0; i < 3; ++i) s_first[i] = next_position();
  }
  __syncthreads();
  int pos = s_first[0], pos1 = s_first[1], pos2 = s_first[2];
  if (pos >= 0) load_records(0, pos);
  if (pos1 >= 0) load_records(1, pos1);
  async_copy_wait();
  __syncthreads();
  if (pos >= 0) fourier_tables(0, rec, pos);
  __syncthreads();

  // Who waits for whom.  Per galaxy i the CTA meets before its columns write
  // (C2(i - 1): every thread has left the rows of i - 1), once in each round of
  // columns and between its columns and its rows (C1(i)).  Before C1(i): the
  // columns of i (reading its Fourier tables and record), the Fourier tables
  // of i + 1 (buffer (i + 1) & 1,
  // last read before C1(i - 1); from the record of i + 1, loaded before
  // C1(i - 1)), after C2(i - 1) the real-space terms of i, and the record of
  // i + 2 (the buffer of i - 1, last read before C1(i - 1)).  The rows use no
  // record: what they need of it is in registers.
  int b3 = 0;
  for (int buf = 0; pos >= 0; buf ^= 1) {
    const GalaxyRecord* const r = rec + b3 * C::RECS;
    const int b3n = b3 == 2 ? 0 : b3 + 1;
    const bool work = r->ok != 0;   // uniform
    const float* pc = p.pcoef + ((size_t)first + pos) * PCOEF;
    const DevPsf& ps = p.psfs[work ? r->psf : 0];
    const float2* const psf_hat = ps.spec[B];
    const int k_eig = EIG ? ps.k_eig : 0;
    const int kp = ps.k, nrt1 = work ? r->nrc * kp : 0, nrt = nrt1 + (COMP && work ? r[1].nrc * kp : 0);
    const int64_t off = r->off;
    [[maybe_unused]] const int64_t gal = r->gal;
    if (pos2 >= 0) load_records(b3n == 2 ? 0 : b3n + 1, pos2);
    int pos3 = -1;
    if (tid == 0) pos3 = next_position();
    [[maybe_unused]] const float* const dat = (LOSS && work) ? (p.dptr ? p.dptr[gal] : p.data + off) : nullptr;
    if constexpr (LOSS) {
      // the data patch's lines, on their way to L2
      if (work)
        for (int i = tid; i < N * N / 32; i += THREADS) prefetch_l2(dat + 32 * i);
    }

    // row-pair inputs, [p][k]: the patch itself, or, when adding to what the
    // patch holds, this CTA's slice of the workspace scratch
    float2* const zbuf = p.accumulate ? p.scratch256 + (size_t)blockIdx.x * (N / 2) * N
                                      : reinterpret_cast<float2*>(p.out + off);
    // Lanczos and adding to the patch: the Fourier part of a galaxy with
    // real-space terms stays there until they are convolved (the model is added
    // to the patch as a whole)
    const bool park = LZ && p.accumulate != 0 && nrt > 0;

    // ---- Steps 5-6 on the bins l = j + m T of each of the group's columns, Step 7a ----
    float2 v[16];
    if (work) {
      const float2* const py = pys + buf * HALF;
      const float4* const fc = fcs + buf * C::RECS * KMAX;
#pragma unroll 1
      for (int cc = 0; cc < ROUNDS; ++cc) {
        const int col = GROUPS * cc + f;   // column nu = col / N
        const float2* ph = psf_hat + col * LS + j;
        const float nu = (float)col * INV_N;
        const float2 pxk = pxs[buf * NP + col];
        if (EIG && k_eig) {
          eigen_bins(ph, PSF_ELEMS, k_eig, pc, [](int m) { return m * T; }, v);
        } else {
#pragma unroll
          for (int m = 0; m < 16; ++m) v[m] = __ldg(ph + m * T);
        }
        float2 s[8];
#pragma unroll
        for (int k = 0; k < 8; ++k) s[k] = make_float2(0.0f, 0.0f);
        mixture16(fc, r->nf, r->s11, 2.0f * r->s12, r->s22, nu, (float)j * INV_N, s);
        if constexpr (COMP)
          mixture16(fc + r->nf, r[1].nf, r[1].s11, 2.0f * r[1].s12, r[1].s22, nu, (float)j * INV_N, s);
#pragma unroll
        for (int m = 0; m < 16; ++m) {
          const int l = j + m * T;
          const float2 e = m < 8 ? cmul(pxk, py[l]) : cmulc(pxk, py[N - l]);
          v[m] = cscale(cmul(v[m], e), (m & 1) ? s[m >> 1].y : s[m >> 1].x);
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
        if (cc == 0) __syncthreads();   // C2 of the previous galaxy
        float2* const wr = W + (cc & 1) * GROUPS * CS + f * CS + j;
        dft16<+1>(v);
#pragma unroll
        for (int k1 = 0; k1 < 16; ++k1) wr[k1 * EX] = k1 ? cmul(v[at16(k1)], tw[k1 - 1]) : v[0];
        __syncthreads();   // this round's first passes are done (and the reads of the round before last)
        // second pass: thread (t, c) of column k = 16 cc + c, c along the half-warp
        const int t = f, k = GROUPS * cc + j;
        const float2* const rd = W + (cc & 1) * GROUPS * CS + j * CS + t * EX;
#pragma unroll
        for (int i = 0; i < 16; ++i) v[i] = rd[i];
        dft16<+1>(v);
        // rows n = t + 16 k2: pairs (p, p + N/2) are k2, k2 + 8
        float2* const zk = zbuf + zpos(t, k);
        float2* const zm = zbuf + zpos(t, k ? N - k : N / 2);
#pragma unroll
        for (int k2 = 0; k2 < 8; ++k2) {
          const float2 A = v[at16(k2)], Bv = v[at16(k2 + 8)];
          zk[16 * k2 * (N / 2)] = k ? make_float2(A.x - Bv.y, A.y + Bv.x) : make_float2(A.x, Bv.x);
          zm[16 * k2 * (N / 2)] = k ? make_float2(A.x + Bv.y, Bv.x - A.y) : make_float2(A.y, Bv.y);
        }
      }
      // the real-space terms, from the last threads down (the first ones have
      // more of the Fourier tables)
      const int nr2 = real_terms_padded(nrt);
      for (int t = THREADS - 1 - tid; t < nr2; t += THREADS) {
        if (t < nrt1) real_term(r[0], ps.mog, (EIG && k_eig) ? pc + 8 : nullptr, kp, N, t, &rt);
        else if (COMP && t < nrt) real_term(r[1], ps.mog, nullptr, kp, N, t - nrt1, &rt, t);
        else real_term_zero(t, &rt);
      }
      if constexpr (LZ) {
        if (tid < 16) s_lzw[buf][tid] = p.lzw[((size_t)first + pos) * 16 + tid];
      }
    } else {
      __syncthreads();   // C2
    }
    if (pos1 >= 0) fourier_tables(buf ^ 1, rec + b3n * C::RECS, pos1);
    if (tid == 0) s_pos[buf] = pos3;
    async_copy_wait();
    __syncthreads();   // C1
    pos3 = s_pos[buf];
    if constexpr (LOSS) {
      if (tid == 0) {
        write_chi2();   // the previous galaxy's
        if (!work) p.chi2[gal] = __int_as_float(0x7fc00000);   // NaN: a galaxy that is skipped
      }
    }

    // ---- Step 7b: row pairs, inputs Z[k], k = j + m T; Step 8 ----
    if (work) {
      [[maybe_unused]] float* const mdl = (LOSS && p.model) ? p.model + off : nullptr;
      [[maybe_unused]] const float iv = LOSS ? p.ivar[gal] : 0.0f;
      [[maybe_unused]] float chi = 0.0f;
#pragma unroll 1
      for (int rr = 0; rr < ROUNDS; ++rr) {
        const int pr = GROUPS * rr + f;   // rows pr and pr + N/2
#pragma unroll
        for (int m = 0; m < 16; ++m) v[m] = __ldcg(&zbuf[zpos(pr, j + m * T)]);
        float2* const w = W + f * RSTR;
        __syncwarp();   // the group's two rows of the round before have been stored
        fft16<N, +1>(
            tw, v, [&](int k1) { return w + k1 * EX + j; }, [&](int q, int i) { return w + j * EX + i; });
        // Pixel x is staged at x ^ cx ^ 4 [bit 5 of x]: the scalar stores of the
        // warp's two groups take different banks, and so do the lanes that
        // read runs of 8 pixels as two 16-byte pieces.
        float* const orow = reinterpret_cast<float*>(w);
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
        float* const dst = (park ? reinterpret_cast<float*>(zbuf) : p.out + off) + (size_t)pr * N;
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
            else store8(dst + h * (N / 2) * N + x0, ov, p.accumulate != 0 && !park);
          }
        }
        if constexpr (LOSS) {
          // every two rounds (32 row pairs) have a sum per warp: the order in
          // which the cluster kernel, a CTA for each 32, adds them
          if (rr & 1) {
            for (int o2 = 16; o2 > 0; o2 >>= 1) chi += __shfl_xor_sync(0xffffffffu, chi, o2);
            if ((tid & 31) == 0) s_chi[LOSS ? buf : 0][(rr >> 1) * WARPS + (tid >> 5)] = chi;
            chi = 0.0f;
          }
        }
      }
      if constexpr (LOSS) {
        if (tid == 0) {
          chi_gal = gal;
          chi_iv = iv;
          chi_buf = buf;
        }
      }
    }
    if constexpr (LZ) {
      if (nrt > 0) {   // uniform
        __syncthreads();   // the whole Fourier part is in the patch (or parked); W is free
        float* const dst = p.out + off;
        const float* const src = park ? reinterpret_cast<const float*>(zbuf) : dst;
        lanczos_real_strips<N, STRIP, THREADS>(
            rt, nrt, s_lzw[LZ ? buf : 0], reinterpret_cast<float*>(smem), [&](int y, int x0, const float(&acc)[8]) {
              const float4* const d = reinterpret_cast<const float4*>(src + y * N + x0);
              const float4 f0 = d[0], f1 = d[1];   // the Fourier part, written by this CTA
              const float ov[8] = {f0.x + acc[0], f0.y + acc[1], f0.z + acc[2], f0.w + acc[3],
                                   f1.x + acc[4], f1.y + acc[5], f1.z + acc[6], f1.w + acc[7]};
              store8(dst + y * N + x0, ov, park);
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

template <bool LZ, bool EIG, bool LOSS, bool COMP>
static int fwd256_occupancy() {
  const int occ = kernel_occupancy(reinterpret_cast<const void*>(render_fwd256_kernel<LZ, EIG, LOSS, COMP>), THREADS,
                                   Cfg256<COMP>::SMEM);
  return occ < 0 ? occ : (occ < CTAS_PER_SM ? occ : CTAS_PER_SM);
}

template <bool LZ, bool EIG, bool LOSS = false, bool COMP = false>
static cudaError_t launch_fwd256(const RenderParams& p, int num_sms, int ctas_per_sm, cudaStream_t s) {
  const int occ = fwd256_occupancy<LZ, EIG, LOSS, COMP>();
  if (occ < 0) return cudaErrorInvalidConfiguration;
  // the accumulate mode's scratch holds one slice per CTA, CTAS_PER_SM per SM
  const int ctas = (ctas_per_sm > 0 && ctas_per_sm < occ) ? ctas_per_sm : occ;
  render_fwd256_kernel<LZ, EIG, LOSS, COMP><<<persistent_grid(p, ctas, num_sms), THREADS, Cfg256<COMP>::SMEM, s>>>(p);
  return cudaGetLastError();
}

// Few galaxies: a cluster per galaxy (render_fwd256c.cu).  A CTA of this kernel
// takes about 80 us for a galaxy, so below a few hundred galaxies the call takes
// that long however few they are (10: 64 us on the earlier 512-thread CTAs, 30
// on clusters), and up to four rounds of its 304 CTAs the last, partly filled one
// weighs more than the clusters' lower rate: calls of 1000 galaxies on clusters
// 239 us against 269 (Lanczos 325 against 361, composites 304 against 327), of
// 1500 339 against 331 (463 against 452, 436 against 402), of 3000 630 against
// 587 (845 against 764, 817 against 729).
cudaError_t launch_render_fwd256_composite(const RenderParams& p, int num_sms, int ctas_per_sm, cudaStream_t s,
                                           const SideStream* side) {
  return launch_by_count(
      p, few256_render(num_sms), far256_render(num_sms), s, side,
      [&](const RenderParams& q, cudaStream_t qs) { return launch_render_fwd256_small(q, num_sms, qs); },
      [&](const RenderParams& q, cudaStream_t qs) {
        return q.lanczos ? launch_fwd256<true, false, false, true>(q, num_sms, ctas_per_sm, qs)
                         : launch_fwd256<false, false, false, true>(q, num_sms, ctas_per_sm, qs);
      });
}

int render_fwd256_max_ctas(int) { return fwd256_occupancy<false, false, false, false>(); }

cudaError_t launch_render_fwd256(const RenderParams& p, int num_sms, int ctas_per_sm, cudaStream_t s,
                                 const SideStream* side) {
  return launch_by_count(
      p, few256_render(num_sms), far256_render(num_sms), s, side,
      [&](const RenderParams& q, cudaStream_t qs) { return launch_render_fwd256_small(q, num_sms, qs); },
      [&](const RenderParams& q, cudaStream_t qs) {
        if (q.loss)
          return q.eigen ? launch_fwd256<false, true, true>(q, num_sms, ctas_per_sm, qs)
                         : launch_fwd256<false, false, true>(q, num_sms, ctas_per_sm, qs);
        if (q.eigen)
          return q.lanczos ? launch_fwd256<true, true>(q, num_sms, ctas_per_sm, qs)
                           : launch_fwd256<false, true>(q, num_sms, ctas_per_sm, qs);
        return q.lanczos ? launch_fwd256<true, false>(q, num_sms, ctas_per_sm, qs)
                         : launch_fwd256<false, false>(q, num_sms, ctas_per_sm, qs);
      });
}

}  // namespace mog
