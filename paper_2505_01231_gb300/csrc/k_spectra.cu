// k_spectra.cu -- K1: frame, window, real FFT, group centring and S2.
//
// One CTA handles one group of m consecutive frames at a time (persistent loop
// over groups).  For every channel and frame j of the group it
//   1. reads the T samples of the frame (Sec. 3, Eq. 16) from the concatenation
//      carry-over | chunk and multiplies them by the window g_i / sqrt(sum g^2)
//      (Eq. 17; the scale is undone in the finalize step),
//   2. packs them as N = T/2 complex points y_n = x_{2n} + j x_{2n+1} and runs a
//      Stockham autosort FFT with the POSITIVE exponent of Eq. 18 (radix-8/4/2
//      butterflies in registers, ping-pong buffers in shared memory),
//   3. splits the half-length transform into the T/2+1 coefficients
//      X_k = E_k + e^{+2 pi j k/T} O_k of the real frame, and writes them.
// After the m frames it subtracts the group mean of every bin (the centred
// samples of the factorised k-statistics, App. H, Eq. 85), and forms the
// per-group S2 estimate c2 = 1/(m-1) sum_j |dX_jk|^2 (Eq. 32 with y = x*),
// whose sum and sum of squares over groups are accumulated for Eq. 35-36.
#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include <algorithm>

#include "internal.cuh"

namespace ss {
namespace {

__device__ __forceinline__ float2 cadd(float2 a, float2 b) { return make_float2(a.x + b.x, a.y + b.y); }
__device__ __forceinline__ float2 csub(float2 a, float2 b) { return make_float2(a.x - b.x, a.y - b.y); }
__device__ __forceinline__ float2 cmul(float2 a, float2 b) {
  return make_float2(fmaf(a.x, b.x, -a.y * b.y), fmaf(a.x, b.y, a.y * b.x));
}
// multiplication by +j
__device__ __forceinline__ float2 cj(float2 a) { return make_float2(-a.y, a.x); }

// Radix-R DFT with the positive exponent, V_q = sum_r v_r e^{+2 pi j rq/R}.
__device__ __forceinline__ void dft4(float2& v0, float2& v1, float2& v2, float2& v3) {
  const float2 s02 = cadd(v0, v2), d02 = csub(v0, v2);
  const float2 s13 = cadd(v1, v3), d13 = cj(csub(v1, v3));
  v0 = cadd(s02, s13);
  v2 = csub(s02, s13);
  v1 = cadd(d02, d13);
  v3 = csub(d02, d13);
}

template <int R>
__device__ __forceinline__ void dft(float2 (&v)[R]);

template <>
__device__ __forceinline__ void dft<2>(float2 (&v)[2]) {
  const float2 a = v[0];
  v[0] = cadd(a, v[1]);
  v[1] = csub(a, v[1]);
}

template <>
__device__ __forceinline__ void dft<4>(float2 (&v)[4]) {
  dft4(v[0], v[1], v[2], v[3]);
}

template <>
__device__ __forceinline__ void dft<8>(float2 (&v)[8]) {
  // even/odd split: V_q = E_q + w^q O_q, V_{q+4} = E_q - w^q O_q, w = e^{+2 pi j/8}
  float2 e0 = v[0], e1 = v[2], e2 = v[4], e3 = v[6];
  float2 o0 = v[1], o1 = v[3], o2 = v[5], o3 = v[7];
  dft4(e0, e1, e2, e3);
  dft4(o0, o1, o2, o3);
  const float h = 0.70710678118654752f;
  o1 = make_float2((o1.x - o1.y) * h, (o1.x + o1.y) * h);    // * (1 + j)/sqrt 2
  o2 = cj(o2);                                                // * j
  o3 = make_float2((-o3.x - o3.y) * h, (o3.x - o3.y) * h);   // * (-1 + j)/sqrt 2
  v[0] = cadd(e0, o0); v[4] = csub(e0, o0);
  v[1] = cadd(e1, o1); v[5] = csub(e1, o1);
  v[2] = cadd(e2, o2); v[6] = csub(e2, o2);
  v[3] = cadd(e3, o3); v[7] = csub(e3, o3);
}

// Where point i of a frame lies in a shared-memory buffer or coefficient row: its place
// within 16 points is XOR-ed with bits of i, so that the strided stores of the first
// passes (8 points apart, then 8 within 64) fall on distinct banks like the consecutive
// loads.  Blocks of 16 points stay in place.
__device__ __forceinline__ int swz(int i) { return i ^ ((i >> 4) & 7) ^ ((i >> 3) & 8); }

// One Stockham pass: sub-transforms of length Ns are combined R at a time into
// length Ns*R.  x, y: N complex points in shared memory; twp: the pass's twiddles
// (twiddle_angle).
template <int R>
__device__ __forceinline__ void stockham_pass(const float2* __restrict__ x, float2* __restrict__ y,
                                              int N, int Ns, const float2* __restrict__ twp) {
  const int NR = N / R;
  for (int j = threadIdx.x; j < NR; j += blockDim.x) {
    const int k = j & (Ns - 1);
    float2 v[R];
#pragma unroll
    for (int r = 0; r < R; ++r) v[r] = x[swz(j + r * NR)];
    if (Ns > 1) {
#pragma unroll
      for (int r = 1; r < R; ++r) v[r] = cmul(v[r], __ldg(&twp[(r - 1) * Ns + k]));
    }
    dft<R>(v);
    const int base = (j - k) * R + k;
#pragma unroll
    for (int q = 0; q < R; ++q) y[swz(base + q * Ns)] = v[q];
  }
}

__device__ __forceinline__ uint32_t to_tf32(float x) {
  uint32_t t;
  asm("cvt.rna.tf32.f32 %0, %1;" : "=r"(t) : "f"(x));
  return t;
}

// e^{+2 pi j k/T} for k = 0 .. N = T/2 from the entries 0 .. N/2 (w^{N-k} = -conj w^k)
template <class At>
__device__ __forceinline__ float2 split_twiddle(At at, int k, int N) {
  const float2 w = at(2 * k <= N ? k : N - k);
  return 2 * k <= N ? w : make_float2(-w.x, w.y);
}

// Write one bin's row of one K chunk (16 entries) of the Gram operand image:
// the hi and lo parts of the entries, in the K-major core-matrix layout the
// tensor cores read (8 rows x 16 bytes per core matrix, 16-byte entry groups
// 128 bytes apart; the hi block of a row group's chunk is followed by its lo
// block).  `row` is the bin's 16-byte slot in the chunk's first hi matrix.
template <int FMT>
__device__ __forceinline__ void write_gram_row(unsigned char* row, const float (&e)[16]) {
  constexpr uint32_t CB = FMT == kImageGramTF32 ? 512u : 256u;
  if constexpr (FMT == kImageGramF16) {
#pragma unroll
    for (int kg = 0; kg < 2; ++kg) {
      uint32_t hi[4], lo[4];
#pragma unroll
      for (int t = 0; t < 4; ++t) {
        // two entries per conversion (each rounded to nearest, as one at a time)
        const float v0 = e[8 * kg + 2 * t], v1 = e[8 * kg + 2 * t + 1];
        const __half2 h = __floats2half2_rn(v0, v1);
        const float2 hf = __half22float2(h);
        const __half2 l = __floats2half2_rn(v0 - hf.x, v1 - hf.y);
        hi[t] = *reinterpret_cast<const uint32_t*>(&h);
        lo[t] = *reinterpret_cast<const uint32_t*>(&l);
      }
      *reinterpret_cast<uint4*>(row + kg * 128) = make_uint4(hi[0], hi[1], hi[2], hi[3]);
      *reinterpret_cast<uint4*>(row + CB + kg * 128) = make_uint4(lo[0], lo[1], lo[2], lo[3]);
    }
  } else if constexpr (FMT == kImageGramTF32) {
#pragma unroll
    for (int kg = 0; kg < 4; ++kg) {
      uint32_t hi[4], lo[4];
#pragma unroll
      for (int t = 0; t < 4; ++t) {
        hi[t] = to_tf32(e[4 * kg + t]);
        lo[t] = to_tf32(e[4 * kg + t] - __uint_as_float(hi[t]));
      }
      *reinterpret_cast<uint4*>(row + kg * 128) = make_uint4(hi[0], hi[1], hi[2], hi[3]);
      *reinterpret_cast<uint4*>(row + CB + kg * 128) = make_uint4(lo[0], lo[1], lo[2], lo[3]);
    }
  } else {
#pragma unroll
    for (int kg = 0; kg < 2; ++kg) {
      uint32_t hi[4], lo[4];
#pragma unroll
      for (int t = 0; t < 4; ++t) {
        const float v0 = e[8 * kg + 2 * t], v1 = e[8 * kg + 2 * t + 1];
        const __nv_bfloat162 h = __floats2bfloat162_rn(v0, v1);
        const float2 hf = __bfloat1622float2(h);
        const __nv_bfloat162 l = __floats2bfloat162_rn(v0 - hf.x, v1 - hf.y);
        hi[t] = *reinterpret_cast<const uint32_t*>(&h);
        lo[t] = *reinterpret_cast<const uint32_t*>(&l);
      }
      *reinterpret_cast<uint4*>(row + kg * 128) = make_uint4(hi[0], hi[1], hi[2], hi[3]);
      *reinterpret_cast<uint4*>(row + CB + kg * 128) = make_uint4(lo[0], lo[1], lo[2], lo[3]);
    }
  }
}

// Several channels in FP16X3: the row scale of a bin whose largest |d_j|^2 over
// the group is mx2, a power of two that brings sqrt(mx2) below 2^14, within
// [2^-60, 2^60] (1 for a zero bin).
__device__ __forceinline__ float cross_row_scale(float mx2) {
  if (!(mx2 > 0.f)) return 1.f;
  int e;
  frexpf(sqrtf(mx2), &e);  // sqrt(mx2) < 2^e
  return ldexpf(1.f, min(60, max(-60, 14 - e)));
}

// FP16 operand image: the power of two that brings a bin's largest entry (the
// weighted Gram products and ps), bounded by `bound`, below 2^14 (1 for an
// all-zero bin).
__device__ __forceinline__ float f16_row_scale(float bound) {
  if (!(bound > 0.f)) return 1.f;
  int e;
  frexpf(bound, &e);  // bound < 2^e
  return ldexpf(1.f, 14 - e);
}

// Coefficient of bin k of a spectra row (bin 0 at row[0]); with mirror, also its
// conjugate at bin -k (several channels: K2 reads whole rows of signed bins).
__device__ __forceinline__ void put_coef(float2* __restrict__ row, int k, int M, float2 d,
                                         int mirror) {
  row[k] = d;
  if (mirror && k > 0 && k < M) row[-k] = make_float2(d.x, -d.y);
}

template <int DTYPE>
__device__ __forceinline__ float load_sample(const SampleSource& s, int c, long long idx) {
  if (idx < s.carry_n) {
    const long long o = (long long)c * s.carry_stride + idx;
    if (DTYPE == SS_F32) return __ldg(static_cast<const float*>(s.carry) + o);
    return (float)__ldg(static_cast<const short*>(s.carry) + o);
  }
  const long long o = (long long)c * s.chunk_stride + (idx - s.carry_n);
  if (DTYPE == SS_F32) return __ldg(static_cast<const float*>(s.chunk) + o);
  return (float)__ldg(static_cast<const short*>(s.chunk) + o);
}

// First-order spectrum of one group (Sec. 4, App. G): the group mean of the
// zero-frequency coefficient (divided by sum g at finalize); its sum and sums of
// squares over the CTA's groups.  Called by the thread that centres bin 0.
__device__ __forceinline__ void add_s1(float* s1, float2 mean) {
  s1[0] += mean.x;
  s1[1] += mean.y;
  s1[2] = fmaf(mean.x, mean.x, s1[2]);
  s1[3] = fmaf(mean.y, mean.y, s1[3]);
}

// Centre bin k over the group's m frames (subtract the mean, the samples of the
// factorised k-statistics, App. H, Eq. 85), store the centred coefficients,
// add the per-group S2 estimate c2 = 1/(m-1) sum_j |d_j|^2 (Eq. 32) to the
// CTA's float32 sums, and, with an operand image, write the bin's weighted Gram
// products (diagonal chunks sqrt(w_jj r) |d_j|^2, then the pairs j < j' in
// lexicographic order, sqrt(4(m-1) r) Re(d_j d_j'*), 16 per chunk, zero-padded)
// and its ps value.  fetch(j) gives frame j's coefficient, store(j, d) keeps the
// centred one.
template <int FMT, class Fetch, class Store>
__device__ __forceinline__ void centre_bin(int k, bool valid, float2 mean, int m, int c, int g,
                                           int Mp, const OperandImage& oi, Fetch fetch,
                                           Store store, float* s2sum, float* s2sq, float pref2) {
  float p = 0.f;
  if constexpr (FMT == kImageNone) {
    float mx = 0.f;  // max_j |d_j|^2 (several channels in FP16X3: the bin's row scale)
    for (int j = 0; j < m; ++j) {
      const float2 d = valid ? csub(fetch(j), mean) : make_float2(0.f, 0.f);
      store(j, d);
      p = fmaf(d.x, d.x, fmaf(d.y, d.y, p));
      mx = fmaxf(mx, fmaf(d.x, d.x, d.y * d.y));
    }
    if (oi.rmax) oi.rmax[(long long)c * oi.chan_rmax + (long long)g * Mp + k] = cross_row_scale(mx);
  } else {
    float dr[kMaxGramM], di[kMaxGramM];
    float mx = 0.f;  // max_j |d_j|^2
    for (int j = 0; j < m; ++j) {
      const float2 d = valid ? csub(fetch(j), mean) : make_float2(0.f, 0.f);
      store(j, d);
      dr[j] = d.x;
      di[j] = d.y;
      const float pj = fmaf(d.x, d.x, d.y * d.y);
      p += pj;
      mx = fmaxf(mx, pj);
    }
    const float sc =
        FMT == kImageGramF16 ? f16_row_scale(fmaxf(fmaxf(oi.sd, oi.so) * mx, oi.sp * p)) : 1.f;
    const float sd = oi.sd * sc, so = oi.so * sc, sps = oi.sp * p * sc;
    const int npair = m * (m - 1) / 2;
    int pj = 0, pk = 1;  // next off-diagonal pair (j, j'), lexicographic
    if (FMT == kImageGramF32) {
      if (k < oi.img_bins) {
        float* e = static_cast<float*>(oi.img) + (size_t)g * oi.rows * Mp + k;
        const int nd = npair + 1;
        for (int j = 0; j < m; ++j) {
          for (int q = j + 1; q < m; ++q, e += Mp) *e = so * fmaf(dr[j], dr[q], di[j] * di[q]);
        }
        *e = sps;
        e += Mp;
        for (int j = 0; j < m; ++j, e += Mp) *e = sd * fmaf(dr[j], dr[j], di[j] * di[j]);
        for (int r = nd + m; r < oi.rows; ++r, e += Mp) *e = 0.f;
      }
    } else if (k < oi.img_bins) {  // rows the tensor-core S4 reads
      constexpr int kChunkBytes = FMT == kImageGramTF32 ? 1024 : 512;  // 2 CB
      unsigned char* rbase = static_cast<unsigned char*>(oi.img) + (size_t)c * oi.chan_bytes +
                             (size_t)g * oi.group_bytes + (size_t)(k >> 3) * oi.rg_bytes +
                             (k & 7) * 16;
      for (int ch = 0; ch < oi.nkc; ++ch) {
        float e[16];
        if (ch < oi.ndc) {
#pragma unroll
          for (int t = 0; t < 16; ++t) {
            const int j = ch * 16 + t;
            e[t] = j < m ? sd * fmaf(dr[j], dr[j], di[j] * di[j]) : 0.f;
          }
        } else {
          const int p0 = (ch - oi.ndc) * 16;
#pragma unroll
          for (int t = 0; t < 16; ++t) {
            if (p0 + t < npair) {
              e[t] = so * fmaf(dr[pj], dr[pk], di[pj] * di[pk]);
              if (++pk == m) {
                ++pj;
                pk = pj + 1;
              }
            } else {
              e[t] = p0 + t == npair ? sps : 0.f;  // ps after the pairs (negated with them)
            }
          }
        }
        write_gram_row<FMT>(rbase + ch * kChunkBytes, e);
      }
      if (FMT == kImageGramF16)  // exact: a power of two
        oi.rsc[(long long)c * oi.chan_rsc + (long long)g * Mp + k] = 1.f / sc;
    }
  }
  if (valid && s2sum) {
    const float c2 = p * pref2;
    s2sum[k] += c2;
    s2sq[k] = fmaf(c2, c2, s2sq[k]);
  }
}

// Add the CTA's float32 sums of S2 (and S1) over its last groups to the float64
// accumulators and clear them.  Each thread flushes the bins it centres (bin k
// belongs to thread k mod blockDim.x; S1 to thread 0), so no barrier is needed.
__device__ __forceinline__ void flush_k1_sums(int C, int M, const int* __restrict__ s2_auto,
                                              double* __restrict__ acc2, int n_s2, float* s2sum,
                                              float* s2sq, float (*s1s)[4], double* acc1) {
  const long long plane = (long long)n_s2 * M;
  for (int c = 0; c < C; ++c) {
    const int ia = s2_auto[c];
    if (ia < 0) continue;
    for (int k = threadIdx.x; k < M; k += blockDim.x) {
      atomicAdd(acc2 + 0 * plane + (long long)ia * M + k, widen(s2sum[c * M + k]));
      atomicAdd(acc2 + 2 * plane + (long long)ia * M + k, widen(s2sq[c * M + k]));
      s2sum[c * M + k] = 0.f;
      s2sq[c * M + k] = 0.f;
    }
  }
  if (threadIdx.x == 0)
    for (int c = 0; c < C; ++c)
      for (int q = 0; q < 4; ++q) {
        if (acc1) atomicAdd(acc1 + q * C + c, widen(s1s[c][q]));
        s1s[c][q] = 0.f;
      }
}

template <int DTYPE, int FMT>
__global__ void __launch_bounds__(kThreadsK1)
k1_spectra(SampleSource src, long long sample0, int G, int C, int T, int m, int M, int Mp,
           const float* __restrict__ win, const float2* __restrict__ tw,
           SpecRows sp, const int* __restrict__ s2_auto,
           double* __restrict__ acc2, int n_s2, float pref2, OperandImage oi,
           double* __restrict__ acc1) {
  extern __shared__ float4 smem_raw[];
  const int N = T / 2;
  float2* bufA = reinterpret_cast<float2*>(smem_raw);
  float2* bufB = bufA + N;
  float2* gsum = bufB + N;                                        // [M]
  float* s2sum = reinterpret_cast<float*>(gsum + M);             // [C][M]
  float* s2sq = s2sum + C * M;                                    // [C][M]

  __shared__ float s1s[4][4];  // per channel: sums of Re, Im, Re^2, Im^2 of S1 (thread 0)
  for (int i = threadIdx.x; i < 2 * C * M; i += blockDim.x) s2sum[i] = 0.f;
  if (threadIdx.x < 16) s1s[threadIdx.x >> 2][threadIdx.x & 3] = 0.f;

  int ngroups = 0;  // groups in the float32 sums since the last flush, all of block cur
  int cur = 0;
  for (int g = blockIdx.x; g < G; g += gridDim.x) {
    if (g / sp.block_groups != cur) {
      if (ngroups)
        flush_k1_sums(C, M, s2_auto, acc2 + cur * sp.block_stride, n_s2, s2sum, s2sq, s1s, acc1);
      ngroups = 0;
      cur = g / sp.block_groups;
    }
    for (int c = 0; c < C; ++c) {
      float2* grow = sp.rows + (long long)c * sp.chan_stride + (long long)g * m * sp.stride;
      for (int k = threadIdx.x; k < M; k += blockDim.x) gsum[k] = make_float2(0.f, 0.f);
      for (int j = 0; j < m; ++j) {
        const long long s0 = sample0 + ((long long)g * m + j) * T;
        __syncthreads();  // bufA is free (previous frame's post-processing done)
        for (int n = threadIdx.x; n < N; n += blockDim.x) {
          const float x0 = load_sample<DTYPE>(src, c, s0 + 2 * n);
          const float x1 = load_sample<DTYPE>(src, c, s0 + 2 * n + 1);
          bufA[swz(n)] = make_float2(x0 * __ldg(&win[2 * n]), x1 * __ldg(&win[2 * n + 1]));
        }
        __syncthreads();
        float2* x = bufA;
        float2* y = bufB;
        int Ns = 1;
        int rem = N;
        const float2* twp = tw + N / 2 + 1;
        while (rem > 1) {
          const int R = fft_radix(rem);
          if (R == 8)
            stockham_pass<8>(x, y, N, Ns, twp);
          else if (R == 4)
            stockham_pass<4>(x, y, N, Ns, twp);
          else
            stockham_pass<2>(x, y, N, Ns, twp);
          if (Ns > 1) twp += (R - 1) * Ns;
          Ns *= R;
          rem /= R;
          __syncthreads();
          float2* t = x; x = y; y = t;
        }
        // x holds Y_n; X_k = 1/2 [(Y_k + Y*_{N-k}) - j w^k (Y_k - Y*_{N-k})], w = e^{+2 pi j/T}
        float2* row = grow + (long long)j * sp.stride;
        for (int k = threadIdx.x; k < M; k += blockDim.x) {
          const float2 yk = x[swz(k == N ? 0 : k)];
          const float2 yr = x[swz(k == 0 ? 0 : N - k)];
          const float2 yc = make_float2(yr.x, -yr.y);
          const float2 s = cadd(yk, yc);
          const float2 wk = split_twiddle([&](int i) { return __ldg(&tw[i]); }, k, N);
          const float2 wd = cmul(wk, csub(yk, yc));
          const float2 X = make_float2(0.5f * (s.x + wd.y), 0.5f * (s.y - wd.x));
          row[k] = X;
          gsum[k] = cadd(gsum[k], X);
        }
      }
      // centre each bin over the group and form the per-group S2 estimate; with an
      // operand image, also write the split tensor-core operands chunk by chunk
      const float inv_m = 1.0f / (float)m;
      const int ia = s2_auto[c];
      for (int k = threadIdx.x; k < Mp; k += blockDim.x) {
        const bool valid = k < M;
        const float2 mean = valid ? make_float2(gsum[k].x * inv_m, gsum[k].y * inv_m)
                                  : make_float2(0.f, 0.f);
        if (k == 0) add_s1(s1s[c], mean);
        centre_bin<FMT>(
            k, valid, mean, m, c, g, Mp, oi,
            [&](int j) { return grow[(long long)j * sp.stride + k]; },
            [&](int j, float2 d) { put_coef(grow + (long long)j * sp.stride, k, M, d, sp.mirror); },
            ia >= 0 ? s2sum + c * M : nullptr, ia >= 0 ? s2sq + c * M : nullptr, pref2);
      }
    }
    if (++ngroups == kMaxFp32Groups) {
      flush_k1_sums(C, M, s2_auto, acc2 + cur * sp.block_stride, n_s2, s2sum, s2sq, s1s, acc1);
      ngroups = 0;
    }
  }
  // the CTA's remaining float32 partial sums into the float64 accumulators
  if (ngroups)
    flush_k1_sums(C, M, s2_auto, acc2 + cur * sp.block_stride, n_s2, s2sum, s2sq, s1s, acc1);
}

// The points n, n + 1 (n even) of a row as one 16-byte store (they stay a pair under swz)
__device__ __forceinline__ void put_pair(float2* row, int n, float4 v) {
  const int p = swz(n);
  if (p & 1) v = make_float4(v.z, v.w, v.x, v.y);
  *reinterpret_cast<float4*>(row + (p & ~1)) = v;
}

// Stockham pass over a batch of FB frames of N points (frame f at x + f sx, its
// output at y + f sy); all threads share the FB * N/R butterflies of the pass.
template <int R>
__device__ __forceinline__ void stockham_pass_batch(const float2* __restrict__ x,
                                                    float2* __restrict__ y, int N, int Ns,
                                                    const float2* __restrict__ twp, int FB,
                                                    int sx, int sy) {
  const int NR = N / R;
  const int lg = __ffs(NR) - 1;  // NR is a power of two
  for (int idx = threadIdx.x; idx < FB * NR; idx += blockDim.x) {
    const int f = idx >> lg, j = idx & (NR - 1);
    const float2* xf = x + f * sx;
    float2* yf = y + f * sy;
    const int k = j & (Ns - 1);
    float2 v[R];
#pragma unroll
    for (int r = 0; r < R; ++r) v[r] = xf[swz(j + r * NR)];
    if (Ns > 1) {
#pragma unroll
      for (int r = 1; r < R; ++r) v[r] = cmul(v[r], twp[(r - 1) * Ns + k]);
    }
    dft<R>(v);
    const int base = (j - k) * R + k;
#pragma unroll
    for (int q = 0; q < R; ++q) yf[swz(base + q * Ns)] = v[q];
  }
}

// K1: with bin k's m coefficients in shared memory (frame j's at col[j * cs], the
// thread's own): subtract the bin's group mean (the centred samples of the factorised
// k-statistics, App. H, Eq. 85), write the centred column to the spectra (with store),
// and, with an operand image, the bin's weighted Gram products and its ps value.  Adds
// the group's S1 (s1, if any) and returns sum_j |d_j|^2.
template <int FMT>
__device__ __forceinline__ float centre_column(float2* col, int cs, float2* __restrict__ grow,
                                               int row_stride, int mirror, int store, int k, int c,
                                               int g, int m, int M, int Mp,
                                               const OperandImage& oi, float* s1) {
  const float inv_m = 1.0f / (float)m;
  const bool valid = k < M;
  float2 mean = make_float2(0.f, 0.f);
  if (valid) {
    for (int j = 0; j < m; ++j) mean = cadd(mean, col[j * cs]);
    mean = make_float2(mean.x * inv_m, mean.y * inv_m);
  }
  if (k == 0 && s1) add_s1(s1, mean);
  float p = 0.f, mx = 0.f;  // sum and max over j of |d_j|^2
  for (int j = 0; j < m; ++j) {
    const float2 d = valid ? csub(col[j * cs], mean) : make_float2(0.f, 0.f);
    col[j * cs] = d;
    if (store) put_coef(grow + (long long)j * row_stride, k, M, d, mirror);
    const float pj = fmaf(d.x, d.x, d.y * d.y);
    p += pj;
    mx = fmaxf(mx, pj);
  }
  // several channels in FP16X3: the bin's row scale
  if (oi.rmax) oi.rmax[(long long)c * oi.chan_rmax + (long long)g * Mp + k] = cross_row_scale(mx);
  if (FMT == kImageGramF32 && k < oi.img_bins) {
    // the bin's column of entry rows: pairs, ps, diagonal, zeros
    float* e = static_cast<float*>(oi.img) + (size_t)g * oi.rows * Mp + k;
    for (int j = 0; j < m; ++j) {
      const float2 dj = col[j * cs];
#pragma unroll 4
      for (int q = j + 1; q < m; ++q) {
        const float2 dq = col[q * cs];
        *e = oi.so * fmaf(dj.x, dq.x, dj.y * dq.y);
        e += Mp;
      }
    }
    *e = oi.sp * p;
    e += Mp;
    for (int j = 0; j < m; ++j, e += Mp) {
      const float2 dj = col[j * cs];
      *e = oi.sd * fmaf(dj.x, dj.x, dj.y * dj.y);
    }
    for (int r = m * (m + 1) / 2 + 1; r < oi.rows; ++r, e += Mp) *e = 0.f;
  } else if (FMT != kImageNone && k < oi.img_bins) {  // rows the tensor-core S4 reads
    const float sc =
        FMT == kImageGramF16 ? f16_row_scale(fmaxf(fmaxf(oi.sd, oi.so) * mx, oi.sp * p)) : 1.f;
    const float sd = oi.sd * sc, so = oi.so * sc, sps = oi.sp * p * sc;
    // weighted Gram products of the bin in K order, read from the centred column
    const int npair = m * (m - 1) / 2;
    int pj = 0, pk = 1;
    float2 dj = col[0];
    constexpr int kChunkBytes = FMT == kImageGramTF32 ? 1024 : 512;  // 2 CB
    unsigned char* rbase = static_cast<unsigned char*>(oi.img) + (size_t)c * oi.chan_bytes +
                           (size_t)g * oi.group_bytes + (size_t)(k >> 3) * oi.rg_bytes +
                           (k & 7) * 16;
    for (int ch = 0; ch < oi.nkc; ++ch) {
      float e[16];
      if (ch < oi.ndc) {
#pragma unroll
        for (int t = 0; t < 16; ++t) {
          const int j = ch * 16 + t;
          const float2 d = j < m ? col[j * cs] : make_float2(0.f, 0.f);
          e[t] = sd * fmaf(d.x, d.x, d.y * d.y);
        }
      } else {
        const int p0 = (ch - oi.ndc) * 16;
#pragma unroll
        for (int t = 0; t < 16; ++t) {
          if (p0 + t < npair) {
            const float2 d2 = col[pk * cs];
            e[t] = so * fmaf(dj.x, d2.x, dj.y * d2.y);
            if (++pk == m) {
              ++pj;
              pk = pj + 1;
              dj = col[pj * cs];
            }
          } else {
            e[t] = p0 + t == npair ? sps : 0.f;  // ps after the pairs (negated with them)
          }
        }
      }
      write_gram_row<FMT>(rbase + ch * kChunkBytes, e);
    }
    if (FMT == kImageGramF16)  // exact: a power of two
      oi.rsc[(long long)c * oi.chan_rsc + (long long)g * Mp + k] = 1.f / sc;
  }
  return p;
}

// K1, resident forms: the group's m coefficient rows of channel c in shared memory (Xs,
// [m][Mp], swizzled within 16), thread = bin; adds the per-group S2 estimate to the
// CTA's float32 sums.
template <int FMT>
__device__ __forceinline__ void centre_resident(float2* Xs, const SpecRows& sp, int c, int g,
                                                int m, int M, int Mp, const OperandImage& oi,
                                                int ia, float* s2sum, float* s2sq, float* s1,
                                                float pref2) {
  float2* grow = sp.rows + (long long)c * sp.chan_stride + (long long)g * m * sp.stride;
  for (int k = threadIdx.x; k < Mp; k += blockDim.x) {
    const float p = centre_column<FMT>(Xs + swz(k), Mp, grow, sp.stride, sp.mirror, sp.store, k, c,
                                       g, m, M, Mp, oi, s1);
    if (k < M && ia >= 0) {
      const float c2 = p * pref2;
      s2sum[c * M + k] += c2;
      s2sq[c * M + k] = fmaf(c2, c2, s2sq[c * M + k]);
    }
  }
}

// K1 for groups whose coefficients fit in shared memory: the group's m frames
// are transformed FB at a time (every Stockham pass covers all FB frames, so a
// frame costs a fraction of the barriers), the coefficients X_jk stay in shared
// memory, and the centred coefficients are written to the spectra once.  The
// passes of a batch alternate between the batch's own coefficient rows and one
// buffer of FB frames (a second buffer would halve FB within the same shared
// memory); the split into X_k reads the last pass's output and writes the rows,
// in place (one thread per pair k, N - k) when the rows hold that output.  Same
// results as k1_spectra; the samples of a batch are contiguous and are read
// with 16-byte (float32) or 8-byte (int16) loads when aligned.
template <int DTYPE, int FMT>
__global__ void __launch_bounds__(kThreadsK1, 3)
k1_spectra_res(SampleSource src, long long sample0, int G, int C, int T, int m, int M, int Mp,
               int FB, const float* __restrict__ win, const float2* __restrict__ tw,
               SpecRows sp, const int* __restrict__ s2_auto,
               double* __restrict__ acc2, int n_s2, float pref2, OperandImage oi,
           double* __restrict__ acc1) {
  extern __shared__ float4 smem_raw[];
  const int N = T / 2;
  float2* buf = reinterpret_cast<float2*>(smem_raw);  // [FB][N]
  float2* Xs = buf + FB * N;                          // [m][Mp]
  float2* tws = Xs + m * Mp;                           // [twiddle_count(T)] twiddles
  float* wins = reinterpret_cast<float*>(tws + twiddle_count(T));  // [T] window / sqrt(sum g^2)
  float* s2sum = wins + T;                             // [C][M]
  float* s2sq = s2sum + C * M;                         // [C][M]
  constexpr int kVec = DTYPE == SS_F32 ? 16 : 8;        // bytes per vector load (4 samples)

  __shared__ float s1s[4][4];  // per channel: sums of Re, Im, Re^2, Im^2 of S1 (thread 0)
  for (int i = threadIdx.x; i < 2 * C * M; i += blockDim.x) s2sum[i] = 0.f;
  if (threadIdx.x < 16) s1s[threadIdx.x >> 2][threadIdx.x & 3] = 0.f;
  for (int i = threadIdx.x; i < T; i += blockDim.x) {
    if (i < twiddle_count(T)) tws[i] = __ldg(&tw[i]);
    wins[i] = __ldg(&win[i]);
  }

  // float32 samples of the next batch, loaded into registers while the current
  // batch is transformed (when the batch is aligned, past the carry-over, and at
  // most kPre vectors per thread)
  constexpr int kPre = 4;
  float4 pre[kPre];
  auto prefetch = [&](int gg, int cc, int jj) -> bool {
    if constexpr (DTYPE != SS_F32) return false;
    const int nq = min(FB, m - jj) * T / 4;
    if (nq > kPre * (int)blockDim.x) return false;
    const long long off = sample0 + ((long long)gg * m + jj) * T - src.carry_n;
    const float4* p4 = reinterpret_cast<const float4*>(
        static_cast<const float*>(src.chunk) + (long long)cc * src.chunk_stride + off);
    if (off < 0 || ((uintptr_t)p4 % 16) != 0) return false;
#pragma unroll
    for (int r = 0; r < kPre; ++r) {
      const int q = threadIdx.x + r * blockDim.x;
      if (q < nq) pre[r] = __ldg(p4 + q);
    }
    return true;
  };
  bool have = blockIdx.x < G && prefetch(blockIdx.x, 0, 0);  // pre holds the batch's samples
  int ngroups = 0;  // groups in the float32 sums since the last flush, all of block cur
  int cur = 0;
  for (int g = blockIdx.x; g < G; g += gridDim.x) {
    if (g / sp.block_groups != cur) {
      if (ngroups)
        flush_k1_sums(C, M, s2_auto, acc2 + cur * sp.block_stride, n_s2, s2sum, s2sq, s1s, acc1);
      ngroups = 0;
      cur = g / sp.block_groups;
    }
    for (int c = 0; c < C; ++c) {
      for (int j0 = 0; j0 < m; j0 += FB) {
        const int nf = min(FB, m - j0);
        const long long s0 = sample0 + ((long long)g * m + j0) * T;  // first sample of the batch
        __syncthreads();  // the buffers are free (previous batch split, previous group centred)
        const long long off = s0 - src.carry_n;
        const char* cbase = static_cast<const char*>(src.chunk) +
                            ((long long)c * src.chunk_stride + off) * (DTYPE == SS_F32 ? 4 : 2);
        if (have) {
#pragma unroll
          for (int r = 0; r < kPre; ++r) {
            const int q = threadIdx.x + r * blockDim.x;
            if (q < nf * T / 4) {
              const int i = (4 * q) & (T - 1), f = (4 * q) / T;
              const float4 w = *reinterpret_cast<const float4*>(wins + i);
              put_pair(Xs + (j0 + f) * Mp, i / 2,
                       make_float4(pre[r].x * w.x, pre[r].y * w.y, pre[r].z * w.z, pre[r].w * w.w));
            }
          }
        } else if (off >= 0 && ((uintptr_t)cbase % kVec) == 0) {
          for (int q = threadIdx.x; q < nf * T / 4; q += blockDim.x) {
            const int i = (4 * q) & (T - 1), f = (4 * q) / T;
            float x0, x1, x2, x3;
            if constexpr (DTYPE == SS_F32) {
              const float4 v = __ldg(reinterpret_cast<const float4*>(cbase) + q);
              x0 = v.x; x1 = v.y; x2 = v.z; x3 = v.w;
            } else {
              const short4 v = __ldg(reinterpret_cast<const short4*>(cbase) + q);
              x0 = v.x; x1 = v.y; x2 = v.z; x3 = v.w;
            }
            const float4 w = *reinterpret_cast<const float4*>(wins + i);
            put_pair(Xs + (j0 + f) * Mp, i / 2,
                     make_float4(x0 * w.x, x1 * w.y, x2 * w.z, x3 * w.w));
          }
        } else {
          for (int q = threadIdx.x; q < nf * N; q += blockDim.x) {
            const int f = q / N, n = q - f * N;
            const long long si = s0 + (long long)f * T + 2 * n;
            Xs[(j0 + f) * Mp + swz(n)] = make_float2(load_sample<DTYPE>(src, c, si) * wins[2 * n],
                                                load_sample<DTYPE>(src, c, si + 1) * wins[2 * n + 1]);
          }
        }
        {  // the next batch: this group's next frames, the next channel or the next group
          int gn = g, cn = c, jn = j0 + FB;
          if (jn >= m) {
            jn = 0;
            if (++cn == C) {
              cn = 0;
              gn += gridDim.x;
            }
          }
          have = gn < G && prefetch(gn, cn, jn);
        }
        __syncthreads();
        float2* rows = Xs + j0 * Mp;
        float2* x = rows;  // the pass input and its frame stride
        float2* y = buf;
        int sx = Mp, sy = N;
        int Ns = 1;
        int rem = N;
        const float2* twp = tws + N / 2 + 1;
        while (rem > 1) {
          const int R = fft_radix(rem);
          if (R == 8)
            stockham_pass_batch<8>(x, y, N, Ns, twp, nf, sx, sy);
          else if (R == 4)
            stockham_pass_batch<4>(x, y, N, Ns, twp, nf, sx, sy);
          else
            stockham_pass_batch<2>(x, y, N, Ns, twp, nf, sx, sy);
          if (Ns > 1) twp += (R - 1) * Ns;
          Ns *= R;
          rem /= R;
          __syncthreads();
          float2* t = x; x = y; y = t;
          const int ts = sx; sx = sy; sy = ts;
        }
        // X_k = 1/2 [(Y_k + Y*_{N-k}) - j w^k (Y_k - Y*_{N-k})], w = e^{+2 pi j/T},
        // Y_N = Y_0: each thread takes a pair k, N - k (k = 0 also gives X_N from
        // Y_0), reads both Y and writes both X, so the split may work in place
        auto split = [&](float2 yk, float2 yr, int k) {
          const float2 yc = make_float2(yr.x, -yr.y);
          const float2 sm = cadd(yk, yc);
          const float2 wd = cmul(split_twiddle([&](int i) { return tws[i]; }, k, N), csub(yk, yc));
          return make_float2(0.5f * (sm.x + wd.y), 0.5f * (sm.y - wd.x));
        };
        const int NH = N / 2 + 1;  // pairs per frame
        for (int idx = threadIdx.x; idx < nf * NH; idx += blockDim.x) {
          const int f = idx / NH, k = idx - f * NH;
          const float2* xf = x + f * sx;
          float2* xr = rows + f * Mp;
          const float2 a = xf[swz(k)], b = xf[swz(k == 0 ? 0 : N - k)];
          xr[swz(k)] = split(a, b, k);
          xr[swz(N - k)] = split(b, a, N - k);
        }
      }
      __syncthreads();  // the group's coefficients are in shared memory
      centre_resident<FMT>(Xs, sp, c, g, m, M, Mp, oi, s2_auto[c], s2sum, s2sq, s1s[c], pref2);
    }
    if (++ngroups == kMaxFp32Groups) {
      flush_k1_sums(C, M, s2_auto, acc2 + cur * sp.block_stride, n_s2, s2sum, s2sq, s1s, acc1);
      ngroups = 0;
    }
  }
  if (ngroups)
    flush_k1_sums(C, M, s2_auto, acc2 + cur * sp.block_stride, n_s2, s2sum, s2sq, s1s, acc1);
}

// One Stockham pass of a warp's own frame (N points in the warp's shared buffer,
// transformed in place): every lane first reads the inputs of its butterflies
// (j = lane + 32 b), the warp synchronises, then each lane writes its outputs.
// N / R <= 32 * (16 / R), i.e. N <= 512: at most 16 points per lane.
template <int R>
__device__ __forceinline__ void warp_stockham_pass(float2* buf, int N, int Ns,
                                                   const float2* __restrict__ twp, int lane) {
  constexpr int kB = 16 / R;  // butterflies per lane
  const int NR = N / R;
  float2 v[kB][R];
#pragma unroll
  for (int b = 0; b < kB; ++b) {
    const int j = lane + 32 * b;
    if (j < NR) {
#pragma unroll
      for (int r = 0; r < R; ++r) v[b][r] = buf[swz(j + r * NR)];
    }
  }
  __syncwarp();
#pragma unroll
  for (int b = 0; b < kB; ++b) {
    const int j = lane + 32 * b;
    if (j < NR) {
      const int k = j & (Ns - 1);
      if (Ns > 1) {
#pragma unroll
        for (int r = 1; r < R; ++r) v[b][r] = cmul(v[b][r], twp[(r - 1) * Ns + k]);
      }
      dft<R>(v[b]);
      const int base = (j - k) * R + k;
#pragma unroll
      for (int q = 0; q < R; ++q) buf[swz(base + q * Ns)] = v[b][q];
    }
  }
  __syncwarp();
}

// K1 with a warp per frame (T <= 1024): the group's coefficients stay resident as
// in k1_spectra_res, but each warp windows, transforms and splits whole frames in
// a buffer of its own, synchronising only itself (no block barrier per pass);
// the block synchronises once per group before and after the centring.
template <int DTYPE, int FMT>
__global__ void __launch_bounds__(kThreadsK1, 2)
k1_spectra_warp(SampleSource src, long long sample0, int G, int C, int T, int m, int M, int Mp,
                const float* __restrict__ win, const float2* __restrict__ tw,
                SpecRows sp, const int* __restrict__ s2_auto,
                double* __restrict__ acc2, int n_s2, float pref2, OperandImage oi,
                double* __restrict__ acc1) {
  extern __shared__ float4 smem_raw[];
  const int N = T / 2;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  constexpr int kWarps = kThreadsK1 / 32;
  float2* Xs = reinterpret_cast<float2*>(smem_raw);  // [m][Mp]
  float2* bufs = Xs + m * Mp;                         // [kWarps][N]
  float2* tws = bufs + kWarps * N;                    // [twiddle_count(T)] twiddles
  float* wins = reinterpret_cast<float*>(tws + twiddle_count(T));  // [T] window / sqrt(sum g^2)
  float* s2sum = wins + T;                            // [C][M]
  float* s2sq = s2sum + C * M;                        // [C][M]
  float2* buf = bufs + warp * N;
  constexpr int kVec = DTYPE == SS_F32 ? 16 : 8;       // bytes per vector load (4 samples)

  __shared__ float s1s[4][4];  // per channel: sums of Re, Im, Re^2, Im^2 of S1 (thread 0)
  for (int i = threadIdx.x; i < 2 * C * M; i += blockDim.x) s2sum[i] = 0.f;
  if (threadIdx.x < 16) s1s[threadIdx.x >> 2][threadIdx.x & 3] = 0.f;
  for (int i = threadIdx.x; i < T; i += blockDim.x) {
    if (i < twiddle_count(T)) tws[i] = __ldg(&tw[i]);
    wins[i] = __ldg(&win[i]);
  }
  __syncthreads();

  int ngroups = 0;  // groups in the float32 sums since the last flush, all of block cur
  int cur = 0;
  for (int g = blockIdx.x; g < G; g += gridDim.x) {
    if (g / sp.block_groups != cur) {
      if (ngroups)
        flush_k1_sums(C, M, s2_auto, acc2 + cur * sp.block_stride, n_s2, s2sum, s2sq, s1s, acc1);
      ngroups = 0;
      cur = g / sp.block_groups;
    }
    for (int c = 0; c < C; ++c) {
      for (int j = warp; j < m; j += kWarps) {
        // the frame's samples times the window, packed as N complex points
        const long long s0 = sample0 + ((long long)g * m + j) * T;
        const long long off = s0 - src.carry_n;
        const char* cbase = static_cast<const char*>(src.chunk) +
                            ((long long)c * src.chunk_stride + off) * (DTYPE == SS_F32 ? 4 : 2);
        if (off >= 0 && ((uintptr_t)cbase % kVec) == 0) {
          for (int q = lane; q < T / 4; q += 32) {
            float x0, x1, x2, x3;
            if constexpr (DTYPE == SS_F32) {
              const float4 v = __ldg(reinterpret_cast<const float4*>(cbase) + q);
              x0 = v.x; x1 = v.y; x2 = v.z; x3 = v.w;
            } else {
              const short4 v = __ldg(reinterpret_cast<const short4*>(cbase) + q);
              x0 = v.x; x1 = v.y; x2 = v.z; x3 = v.w;
            }
            const float4 w = *reinterpret_cast<const float4*>(wins + 4 * q);
            put_pair(buf, 2 * q, make_float4(x0 * w.x, x1 * w.y, x2 * w.z, x3 * w.w));
          }
        } else {
          for (int n = lane; n < N; n += 32)
            buf[swz(n)] = make_float2(load_sample<DTYPE>(src, c, s0 + 2 * n) * wins[2 * n],
                                 load_sample<DTYPE>(src, c, s0 + 2 * n + 1) * wins[2 * n + 1]);
        }
        __syncwarp();
        int Ns = 1, rem = N;
        const float2* twp = tws + N / 2 + 1;
        while (rem > 1) {
          const int R = fft_radix(rem);
          if (R == 8)
            warp_stockham_pass<8>(buf, N, Ns, twp, lane);
          else if (R == 4)
            warp_stockham_pass<4>(buf, N, Ns, twp, lane);
          else
            warp_stockham_pass<2>(buf, N, Ns, twp, lane);
          if (Ns > 1) twp += (R - 1) * Ns;
          Ns *= R;
          rem /= R;
        }
        // X_k = 1/2 [(Y_k + Y*_{N-k}) - j w^k (Y_k - Y*_{N-k})], w = e^{+2 pi j/T}
        float2* xr = Xs + j * Mp;
        for (int k = lane; k < M; k += 32) {
          const float2 yk = buf[swz(k == N ? 0 : k)];
          const float2 yr = buf[swz(k == 0 ? 0 : N - k)];
          const float2 yc = make_float2(yr.x, -yr.y);
          const float2 sm = cadd(yk, yc);
          const float2 wd = cmul(split_twiddle([&](int i) { return tws[i]; }, k, N), csub(yk, yc));
          xr[swz(k)] = make_float2(0.5f * (sm.x + wd.y), 0.5f * (sm.y - wd.x));
        }
        __syncwarp();  // the buffer is free for the warp's next frame
      }
      __syncthreads();  // the group's coefficients are in shared memory
      centre_resident<FMT>(Xs, sp, c, g, m, M, Mp, oi, s2_auto[c], s2sum, s2sq, s1s[c], pref2);
      __syncthreads();  // Xs is free for the next channel or group
    }
    if (++ngroups == kMaxFp32Groups) {
      flush_k1_sums(C, M, s2_auto, acc2 + cur * sp.block_stride, n_s2, s2sum, s2sq, s1s, acc1);
      ngroups = 0;
    }
  }
  if (ngroups)
    flush_k1_sums(C, M, s2_auto, acc2 + cur * sp.block_stride, n_s2, s2sum, s2sq, s1s, acc1);
}

// ---------------------------------------------------------------------------
// K1 for long frames (T >= 1024) whose groups do not fit in shared memory, and for
// power spectra alone.  A 256-thread CTA transforms batches of 2048 complex points
// (FB = 2048 / N consecutive frames of N = T/2 points), one radix-8 butterfly a thread in
// the first pass, whose inputs come straight from global memory (two samples each,
// windowed from shared memory, the next batch's loaded before the current one's passes); the
// other passes go through two swizzled shared-memory buffers, with one barrier each.
//
// kPower: a CTA takes whole groups; thread t owns the bins k = t + 256 s and N - k and
// keeps each bin's running mean and sum of squared deviations over the group's frames
// (Welford's update) in registers, so nothing but the sums leaves the SM.  Else
// the coefficients are written to the spectra as they are, and k1_centre does the rest.
//
// HBM bounds the power form in the end (4 bytes a sample in, nothing out); now it is shared
// memory (LSU 68 %) and issue (68 %).  Measured, S2 alone, T = 2048, m = 16, 2^27 samples:
// 1.11 ms frame by frame with the spectra written, read, centred and written again, now
// 0.257 ms (2.07 TB/s); T = 1024, m = 8, 2^26: 0.123 ms; T = 4096, m = 8, 2^26: 0.144 ms.
// In two kernels, T = 4096, m = 10, int16, 2^24 samples with the FP16 image: 0.246 ms ->
// 0.117 ms (0.044 transform, 0.069 centring); T = 2048, m = 9, 5e6: 0.095 -> 0.042 ms.
constexpr int kFftPoints = 2048;

// one pass of radix R over sub-transforms of length NS, compile-time sizes
template <int R, int NS, int N>
__device__ __forceinline__ void fixed_pass(const float2* __restrict__ x, float2* __restrict__ y,
                                           const float2* __restrict__ twp) {
  constexpr int NR = N / R;
#pragma unroll
  for (int i = 0; i < kFftPoints / R / kThreadsK1; ++i) {
    const int idx = threadIdx.x + i * kThreadsK1;
    const int f = idx / NR, j = idx % NR, k = j % NS;
    const float2* xf = x + f * N;
    float2* yf = y + f * N;
    float2 v[R];
#pragma unroll
    for (int r = 0; r < R; ++r) v[r] = xf[swz(j + r * NR)];
#pragma unroll
    for (int r = 1; r < R; ++r) v[r] = cmul(v[r], twp[(r - 1) * NS + k]);
    dft<R>(v);
    const int base = (j - k) * R + k;
#pragma unroll
    for (int q = 0; q < R; ++q) yf[swz(base + q * NS)] = v[q];
  }
}

// One bin over a group's frames: running mean and sum of squared deviations.
struct Welford {
  float2 mean;
  float m2;
  __device__ __forceinline__ void clear() {
    mean = make_float2(0.f, 0.f);
    m2 = 0.f;
  }
  __device__ __forceinline__ void add(float2 x, float inv_n) {
    const float2 d = csub(x, mean);
    mean = make_float2(fmaf(d.x, inv_n, mean.x), fmaf(d.y, inv_n, mean.y));
    const float2 e = csub(x, mean);
    m2 = fmaf(d.x, e.x, fmaf(d.y, e.y, m2));
  }
};

template <int DTYPE, int N, bool kPower>
__global__ void __launch_bounds__(kThreadsK1, kPower && N == 2048 ? 2 : 3)  // registers
k1_fft(SampleSource src, long long sample0, int G, int m, const float* __restrict__ win,
       const float2* __restrict__ tw, SpecRows sp, const int* __restrict__ s2_auto,
       double* __restrict__ acc2, int n_s2, float pref2, double* __restrict__ acc1, int C) {
  constexpr int T = 2 * N, M = N + 1, FB = kFftPoints / N, NR = N / 8;
  constexpr int kSlots = N / 2 / kThreadsK1;  // bin pairs (k, N - k) of a thread
  extern __shared__ float4 smem_raw[];
  float2* bufA = reinterpret_cast<float2*>(smem_raw);
  float2* bufB = bufA + kFftPoints;
  float2* tws = bufB + kFftPoints;          // [twiddle_count(T)]
  float2* wins = tws + twiddle_count(T);     // [N] pairs of the window
  const int tid = threadIdx.x;
  const int c = blockIdx.y;
  for (int i = tid; i < twiddle_count(T); i += kThreadsK1) tws[i] = __ldg(&tw[i]);
  for (int i = tid; i < N; i += kThreadsK1)
    wins[i] = __ldg(reinterpret_cast<const float2*>(win) + i);
  const int pf = tid / NR, pj = tid % NR;  // frame and butterfly of the first pass

  // samples 2 (pj + r NR), + 1 of frame f0 + pf (of nf frames from f0 on)
  auto load = [&](long long f0, int nf, float2 (&v)[8]) {
    const long long s0 = sample0 + (f0 + pf) * T + 2 * pj;
    const long long off = s0 - src.carry_n;
    constexpr int kVec = DTYPE == SS_F32 ? 8 : 4;  // bytes of two samples
    const char* p = static_cast<const char*>(src.chunk) +
                    ((long long)c * src.chunk_stride + off) * (DTYPE == SS_F32 ? 4 : 2);
    if (pf >= nf) {
#pragma unroll
      for (int r = 0; r < 8; ++r) v[r] = make_float2(0.f, 0.f);
    } else if (off >= 0 && (uintptr_t)p % kVec == 0) {
#pragma unroll
      for (int r = 0; r < 8; ++r) {
        if constexpr (DTYPE == SS_F32) {
          v[r] = __ldg(reinterpret_cast<const float2*>(p) + r * NR);
        } else {
          const short2 q = __ldg(reinterpret_cast<const short2*>(p) + r * NR);
          v[r] = make_float2((float)q.x, (float)q.y);
        }
      }
    } else {
#pragma unroll
      for (int r = 0; r < 8; ++r)
        v[r] = make_float2(load_sample<DTYPE>(src, c, s0 + 2 * r * NR),
                           load_sample<DTYPE>(src, c, s0 + 2 * r * NR + 1));
    }
  };
  // the batch's transforms from v; the result is in the returned buffer after a barrier
  auto transform = [&](float2 (&v)[8]) -> const float2* {
#pragma unroll
    for (int r = 0; r < 8; ++r) {
      const float2 w = wins[pj + r * NR];
      v[r] = make_float2(v[r].x * w.x, v[r].y * w.y);
    }
    dft<8>(v);
#pragma unroll
    for (int q = 0; q < 8; ++q) bufA[pf * N + swz(8 * pj + q)] = v[q];
    __syncthreads();
    const float2* t2 = tws + N / 2 + 1;  // NS = 8
    fixed_pass<8, 8, N>(bufA, bufB, t2);
    __syncthreads();
    const float2* t3 = t2 + 7 * 8;  // NS = 64
    if constexpr (N == 512) {
      fixed_pass<8, 64, N>(bufB, bufA, t3);
      __syncthreads();
      return bufA;
    } else if constexpr (N == 1024) {
      fixed_pass<4, 64, N>(bufB, bufA, t3);
      __syncthreads();
      fixed_pass<4, 256, N>(bufA, bufB, t3 + 3 * 64);
      __syncthreads();
      return bufB;
    } else {
      fixed_pass<8, 64, N>(bufB, bufA, t3);
      __syncthreads();
      fixed_pass<4, 512, N>(bufA, bufB, t3 + 7 * 64);
      __syncthreads();
      return bufB;
    }
  };
  // X_k of Y_k and Y_{N-k} (see k1_spectra_res)
  auto split = [&](float2 yk, float2 yr, float2 wk) {
    const float2 yc = make_float2(yr.x, -yr.y);
    const float2 sm = cadd(yk, yc);
    const float2 wd = cmul(wk, csub(yk, yc));
    return make_float2(0.5f * (sm.x + wd.y), 0.5f * (sm.y - wd.x));
  };
  // The buffer the result lies in is written again no earlier than after the next
  // batch's first barrier (N = 512: its first pass writes the result's buffer, so the
  // split ends with a barrier of its own).
  float2 pre[8];
  if constexpr (!kPower) {
    const long long frames = (long long)G * m, nb = (frames + FB - 1) / FB;
    float2* base = sp.rows + (long long)c * sp.chan_stride;
    long long b = blockIdx.x;
    if (b < nb) load(b * FB, (int)min((long long)FB, frames - b * FB), pre);
    for (; b < nb; b += gridDim.x) {
      const int nf = (int)min((long long)FB, frames - b * FB);
      float2 v[8];
#pragma unroll
      for (int r = 0; r < 8; ++r) v[r] = pre[r];
      const long long bn = b + gridDim.x;
      if (bn < nb) load(bn * FB, (int)min((long long)FB, frames - bn * FB), pre);
      if (b == blockIdx.x) __syncthreads();  // the twiddles are in shared memory
      const float2* Y = transform(v);
#pragma unroll
      for (int f = 0; f < FB; ++f) {
        if (f < nf) {
          const float2* y = Y + f * N;
          float2* row = base + (b * FB + f) * (long long)sp.stride;
#pragma unroll
          for (int s = 0; s < kSlots; ++s) {
            const int k = tid + s * kThreadsK1;
            const float2 a = y[swz(k)], bb = y[swz(k == 0 ? 0 : N - k)];
            const float2 wk = tws[k];
            row[k] = split(a, bb, wk);
            row[N - k] = split(bb, a, make_float2(-wk.x, wk.y));
          }
          if (tid == 0) {
            const float2 a = y[swz(N / 2)];
            row[N / 2] = split(a, a, tws[N / 2]);
          }
        }
      }
      if (N == 512) __syncthreads();
    }
  } else {
    const int ia = s2_auto[c];
    Welford lo[kSlots], hi[kSlots], mid;
    float sum[2 * kSlots + 1], sq[2 * kSlots + 1];  // c2 and its square over the groups
    float s1[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
    for (int i = 0; i < 2 * kSlots + 1; ++i) sum[i] = sq[i] = 0.f;
    auto flush = [&](int blk) {
      const long long plane = (long long)n_s2 * M;
      double* dst = acc2 + blk * sp.block_stride + (long long)ia * M;
      auto put = [&](int k, float a, float b) {
        if (ia < 0) return;
        atomicAdd(dst + k, widen(a));
        atomicAdd(dst + 2 * plane + k, widen(b));
      };
#pragma unroll
      for (int s = 0; s < kSlots; ++s) {
        const int k = tid + s * kThreadsK1;
        put(k, sum[2 * s], sq[2 * s]);
        put(N - k, sum[2 * s + 1], sq[2 * s + 1]);
      }
      if (tid == 0) {
        put(N / 2, sum[2 * kSlots], sq[2 * kSlots]);
        for (int q = 0; q < 4; ++q) {
          if (acc1) atomicAdd(acc1 + q * C + c, widen(s1[q]));
          s1[q] = 0.f;
        }
      }
#pragma unroll
      for (int i = 0; i < 2 * kSlots + 1; ++i) sum[i] = sq[i] = 0.f;
    };
    int g = blockIdx.x, ngroups = 0, cur = 0;
    if (g < G) load((long long)g * m, min(FB, m), pre);
    for (; g < G; g += gridDim.x) {
      if (g / sp.block_groups != cur) {
        if (ngroups) flush(cur);
        ngroups = 0;
        cur = g / sp.block_groups;
      }
#pragma unroll
      for (int s = 0; s < kSlots; ++s) {
        lo[s].clear();
        hi[s].clear();
      }
      mid.clear();
      for (int j0 = 0; j0 < m; j0 += FB) {
        const int nf = min(FB, m - j0);
        float2 v[8];
#pragma unroll
        for (int r = 0; r < 8; ++r) v[r] = pre[r];
        // the next batch: this group's next frames or the CTA's next group's first
        const bool more = j0 + FB < m;
        const long long gn = more ? g : (long long)g + gridDim.x;
        const int jn = more ? j0 + FB : 0;
        if (gn < G) load(gn * m + jn, min(FB, m - jn), pre);
        if (g == (int)blockIdx.x && j0 == 0) __syncthreads();  // the twiddles are there
        const float2* Y = transform(v);
#pragma unroll
        for (int f = 0; f < FB; ++f) {
          if (f < nf) {
            const float2* y = Y + f * N;
            const float inv = 1.0f / (float)(j0 + f + 1);
#pragma unroll
            for (int s = 0; s < kSlots; ++s) {
              const int k = tid + s * kThreadsK1;
              const float2 a = y[swz(k)], bb = y[swz(k == 0 ? 0 : N - k)];
              const float2 wk = tws[k];
              lo[s].add(split(a, bb, wk), inv);
              hi[s].add(split(bb, a, make_float2(-wk.x, wk.y)), inv);
            }
            if (tid == 0) {
              const float2 a = y[swz(N / 2)];
              mid.add(split(a, a, tws[N / 2]), inv);
            }
          }
        }
        if (N == 512) __syncthreads();
      }
      auto add = [&](int i, float m2) {
        const float c2 = m2 * pref2;
        sum[i] += c2;
        sq[i] = fmaf(c2, c2, sq[i]);
      };
#pragma unroll
      for (int s = 0; s < kSlots; ++s) {
        add(2 * s, lo[s].m2);
        add(2 * s + 1, hi[s].m2);
      }
      add(2 * kSlots, mid.m2);
      if (tid == 0) add_s1(s1, lo[0].mean);
      if (++ngroups == kMaxFp32Groups) {
        flush(cur);
        ngroups = 0;
      }
    }
    if (ngroups) flush(cur);
  }
}

// Centring of the spectra that k1_fft wrote (they are still in L2): thread = bin of a
// block of 256, with its column of the group's m coefficients staged in shared memory
// (each thread reads and writes its own column only: no barrier); a CTA takes a run of
// groups and keeps its bins' S2 sums in registers.  Splitting the bins over CTAs instead
// of one CTA per group gives 9 times the loads in flight at T = 4096.
template <int FMT>
__global__ void __launch_bounds__(kThreadsK1)
k1_centre(int G, int m, int M, int Mp, int groups_per_cta, SpecRows sp,
          const int* __restrict__ s2_auto, double* __restrict__ acc2, int n_s2, float pref2,
          OperandImage oi, double* __restrict__ acc1, int C) {
  extern __shared__ float4 smem_raw[];
  float2* col = reinterpret_cast<float2*>(smem_raw) + threadIdx.x;  // [m][256]
  const int k = blockIdx.x * kThreadsK1 + threadIdx.x, c = blockIdx.z;
  if (k >= Mp) return;
  const int g0 = blockIdx.y * groups_per_cta, g1 = min(G, g0 + groups_per_cta);
  float sum = 0.f, sq = 0.f;
  float s1[4] = {0.f, 0.f, 0.f, 0.f};
  const int ia = s2_auto[c];
  int cur = g0 / sp.block_groups;
  auto flush = [&]() {
    if (k >= M || ia < 0) return;
    double* dst = acc2 + cur * sp.block_stride + (long long)ia * M + k;
    atomicAdd(dst, widen(sum));
    atomicAdd(dst + 2 * (long long)n_s2 * M, widen(sq));
    sum = sq = 0.f;
  };
  for (int g = g0; g < g1; ++g) {
    if (g / sp.block_groups != cur) {
      flush();
      cur = g / sp.block_groups;
    }
    float2* grow = sp.rows + (long long)c * sp.chan_stride + (long long)g * m * sp.stride;
    if (k < M) {
#pragma unroll 8
      for (int j = 0; j < m; ++j) col[j * kThreadsK1] = grow[(long long)j * sp.stride + k];
    }
    const float p = centre_column<FMT>(col, kThreadsK1, grow, sp.stride, sp.mirror, 1, k, c, g, m,
                                       M, Mp, oi, s1);
    const float c2 = p * pref2;
    sum += c2;
    sq = fmaf(c2, c2, sq);
  }
  flush();
  if (k == 0 && acc1)
    for (int q = 0; q < 4; ++q) atomicAdd(acc1 + q * C + c, widen(s1[q]));
}

// Cross-channel S2 (Sec. 7, Eq. 47): c2(a_k, b_k*) = 1/(m-1) sum_j da_jk db_jk*
// per group, from the centred spectra K1 wrote.  Thread = (combination, bin);
// blockIdx.y splits the groups; float32 sums per CTA, float64 accumulation.
__global__ void k1_cross_s2(const float2* __restrict__ spec, long long chan_stride, int G, int m,
                            int M, int Mp, const int4* __restrict__ pairs, int groups_per_cta,
                            float pref2, double* __restrict__ acc2, long long plane) {
  const int k = blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= M) return;
  const int4 pr = pairs[blockIdx.z];
  const float2* A = spec + pr.x * chan_stride;
  const float2* B = spec + pr.y * chan_stride;
  const int g0 = blockIdx.y * groups_per_cta;
  const int g1 = min(G, g0 + groups_per_cta);
  float sr = 0.f, si = 0.f, qr = 0.f, qi = 0.f;
  for (int g = g0; g < g1; ++g) {
    float cr = 0.f, ci = 0.f;
    for (int j = 0; j < m; ++j) {
      const long long o = ((long long)g * m + j) * Mp + k;
      const float2 a = A[o], b = B[o];
      cr = fmaf(a.x, b.x, fmaf(a.y, b.y, cr));
      ci = fmaf(a.y, b.x, fmaf(-a.x, b.y, ci));
    }
    cr *= pref2;
    ci *= pref2;
    sr += cr;
    si += ci;
    qr = fmaf(cr, cr, qr);
    qi = fmaf(ci, ci, qi);
  }
  const long long o = (long long)pr.z * M + k;
  atomicAdd(acc2 + o, widen(sr));
  atomicAdd(acc2 + plane + o, widen(si));
  atomicAdd(acc2 + 2 * plane + o, widen(qr));
  atomicAdd(acc2 + 3 * plane + o, widen(qi));
}

}  // namespace

// Dynamic shared memory of the frame-at-a-time K1 for T samples and C channels,
// and its largest value (T = kMaxT, C = kMaxChannels).
constexpr size_t k1_smem(int T, int C) {
  return (size_t)(T / 2) * 2 * sizeof(float2) + (size_t)(T / 2 + 1) * sizeof(float2) +
         (size_t)2 * C * (T / 2 + 1) * sizeof(float);
}
constexpr size_t kK1MaxSmem = k1_smem(kMaxT, kMaxChannels);

// k1_centre keeps a group's columns of 256 bins in shared memory
constexpr size_t kCentreMaxSmem = 160u << 10;

// k1_fft over whole groups (power) or all frames; N = T/2 is 512, 1024 or 2048
template <int DTYPE, bool kPower>
cudaError_t launch_k1_fft(const SampleSource& src, long long sample0, int G, int C, int T, int m,
                          const float* win, const float2* tw, const SpecRows& spec,
                          const int* s2_auto, double* acc2, int n_s2, float pref2, double* acc1,
                          LaunchCache* lc, int nsm, cudaStream_t stream) {
  auto kern = T == 1024   ? k1_fft<DTYPE, 512, kPower>
              : T == 2048 ? k1_fft<DTYPE, 1024, kPower>
                          : k1_fft<DTYPE, 2048, kPower>;
  const size_t smem = (size_t)(2 * kFftPoints + twiddle_count(T) + T / 2) * sizeof(float2);
  const size_t limit = (size_t)(2 * kFftPoints + twiddle_count(kMaxT) + kMaxT / 2) * sizeof(float2);
  int occ = 1;
  cudaError_t e = prepare_kernel((const void*)kern, kThreadsK1, smem, limit, 2048 / kThreadsK1, lc,
                                 kPower ? kSlotK1Power : kSlotK1Fft, &occ);
  if (e != cudaSuccess) return e;
  const int FB = kFftPoints / (T / 2);
  const long long units = kPower ? G : ((long long)G * m + FB - 1) / FB;
  const long long wave = std::max(1, nsm * occ / C);
  kern<<<dim3((unsigned)std::min(units, wave), (unsigned)C), kThreadsK1, smem, stream>>>(
      src, sample0, G, m, win, tw, spec, s2_auto, acc2, n_s2, pref2, acc1, C);
  return cudaGetLastError();
}

template <int FMT>
cudaError_t launch_k1_centre(int G, int C, int m, int M, int Mp, const SpecRows& spec,
                             const int* s2_auto, double* acc2, int n_s2, float pref2,
                             const OperandImage& oi, double* acc1, LaunchCache* lc, int nsm,
                             cudaStream_t stream) {
  const size_t smem = (size_t)m * kThreadsK1 * sizeof(float2);
  if (smem > kCentreMaxSmem) return cudaErrorInvalidValue;
  int occ = 1;
  cudaError_t e = prepare_kernel((const void*)k1_centre<FMT>, kThreadsK1, smem, kCentreMaxSmem, 8, lc,
                                 kSlotK1Centre, &occ);
  if (e != cudaSuccess) return e;
  const int bx = (Mp + kThreadsK1 - 1) / kThreadsK1;
  // about eight CTAs per SM, at most kMaxFp32Groups groups in a float32 sum
  long long gpc = (long long)G * bx * C / (8ll * nsm);
  gpc = std::max(1ll, std::min<long long>(gpc, kMaxFp32Groups));
  while ((G + gpc - 1) / gpc > 65535) ++gpc;  // (more than 4 million groups in a batch)
  k1_centre<FMT><<<dim3((unsigned)bx, (unsigned)((G + gpc - 1) / gpc), (unsigned)C), kThreadsK1,
                   smem, stream>>>(G, m, M, Mp, (int)gpc, spec, s2_auto, acc2, n_s2, pref2, oi,
                                   acc1, C);
  return cudaGetLastError();
}

template <int DTYPE, int FMT>
cudaError_t launch_k1_t(const SampleSource& src, long long sample0, int G, int C, int T, int m,
                        int M, int Mp, const float* win, const float2* tw, const SpecRows& spec,
                        const int* s2_auto, double* acc2, int n_s2,
                        float pref2, const OperandImage& oi, LaunchCache* lc, size_t smem,
                        cudaStream_t stream, double* acc1, int mode) {
  // a group whose coefficients fit beside a batch of FFT buffers stays resident
  const size_t fixed = (size_t)m * Mp * sizeof(float2) + (size_t)2 * C * M * sizeof(float) +
                       (size_t)twiddle_count(T) * sizeof(float2) + (size_t)T * sizeof(float);
  const size_t per_frame = (size_t)(T / 2) * sizeof(float2);  // one buffer of T/2 points
  // kK1Auto: three CTAs per SM with a smaller batch of frames beat two with a
  // larger one (T = 1024, m = 10: 2.59 vs 2.69 ms per step), else the 96 KB
  // budget; kK1Resident96: the 96 KB budget; kK1Frames: frame at a time
  // a warp per frame: the group's coefficients, a buffer of T/2 points per warp;
  // shapes it does not take (T > 1024, or a group beyond 96 KB) use kK1Auto
  const size_t wsmem = fixed + (size_t)(kThreadsK1 / 32) * (T / 2) * sizeof(float2);
  if (mode == kK1Warp && (T > 1024 || wsmem > kK1ResidentBytes)) mode = kK1Auto;
  int nsm = 1, occ = 1;
  cudaError_t e = sm_count(lc, &nsm);
  if (e != cudaSuccess) return e;
  constexpr int kMaxCtas = 2048 / kThreadsK1;
  if (mode == kK1Warp) {
    auto kern = k1_spectra_warp<DTYPE, FMT>;
    e = prepare_kernel((const void*)kern, kThreadsK1, wsmem, kK1ResidentBytes, kMaxCtas, lc,
                       kSlotK1Warp, &occ);
    if (e != cudaSuccess) return e;
    const int rgrid = std::max(1, std::min(G, nsm * occ));
    kern<<<rgrid, kThreadsK1, wsmem, stream>>>(src, sample0, G, C, T, m, M, Mp, win, tw, spec,
                                               s2_auto, acc2, n_s2, pref2, oi, acc1);
    return cudaGetLastError();
  }
  // Long frames: the power spectrum alone from registers; groups that do not fit in
  // shared memory (or kK1Frames) as transform and centring in two kernels.
  if (T >= 1024 && (size_t)m * kThreadsK1 * sizeof(float2) <= kCentreMaxSmem) {
    const bool two = mode == kK1Frames || fixed + per_frame > kK1ResidentBytes;
    if (two || (!spec.store && mode == kK1Auto)) {
      if (!spec.store)
        return launch_k1_fft<DTYPE, true>(src, sample0, G, C, T, m, win, tw, spec, s2_auto, acc2,
                                          n_s2, pref2, acc1, lc, nsm, stream);
      e = launch_k1_fft<DTYPE, false>(src, sample0, G, C, T, m, win, tw, spec, s2_auto, acc2, n_s2,
                                      pref2, acc1, lc, nsm, stream);
      if (e != cudaSuccess) return e;
      return launch_k1_centre<FMT>(G, C, m, M, Mp, spec, s2_auto, acc2, n_s2, pref2, oi, acc1, lc, nsm,
                                   stream);
    }
  }
  const size_t budget = mode == kK1Frames ? 0
                        : (mode == kK1Auto && fixed + per_frame <= kK1ResidentBytes3)
                            ? kK1ResidentBytes3
                            : kK1ResidentBytes;
  if (fixed + per_frame <= budget) {
    const int FB = (int)std::min<size_t>((size_t)m, (budget - fixed) / per_frame);
    const size_t rsmem = fixed + (size_t)FB * per_frame;
    if (rsmem > kK1ResidentBytes) return cudaErrorInvalidValue;  // never: budget <= the limit
    auto kern = k1_spectra_res<DTYPE, FMT>;
    // one wave: as many CTAs as are resident at once
    e = prepare_kernel((const void*)kern, kThreadsK1, rsmem, kK1ResidentBytes, kMaxCtas, lc,
                       budget == kK1ResidentBytes3 ? kSlotK1Res74 : kSlotK1Res96, &occ);
    if (e != cudaSuccess) return e;
    const int rgrid = std::max(1, std::min(G, nsm * occ));
    kern<<<rgrid, kThreadsK1, rsmem, stream>>>(
        src, sample0, G, C, T, m, M, Mp, FB, win, tw, spec, s2_auto, acc2, n_s2,
        pref2, oi, acc1);
    return cudaGetLastError();
  }
  if (smem > kK1MaxSmem) return cudaErrorInvalidValue;
  e = prepare_kernel((const void*)k1_spectra<DTYPE, FMT>, kThreadsK1, smem, kK1MaxSmem, kMaxCtas, lc,
                     kSlotK1Frames, &occ);
  if (e != cudaSuccess) return e;
  k1_spectra<DTYPE, FMT><<<std::min(G, 4 * nsm), kThreadsK1, smem, stream>>>(
      src, sample0, G, C, T, m, M, Mp, win, tw, spec, s2_auto, acc2, n_s2, pref2, oi, acc1);
  return cudaGetLastError();
}

cudaError_t launch_k1_spectra(const SampleSource& src, long long sample0, int G, int C, int T,
                              int m, int M, int Mp, const float* win, const float2* tw,
                              const SpecRows& spec, const int* s2_auto,
                              double* acc2, int n_s2, float pref2, LaunchCache* lc, cudaStream_t stream,
                              const OperandImage& oi, double* acc1, int mode) {
  if (G <= 0) return cudaSuccess;
  if (mode < kK1Auto || mode >= kK1Modes) return cudaErrorInvalidValue;
  const size_t smem = k1_smem(T, C);
  const bool f32 = src.dtype == SS_F32;
#define K1_ARGS src, sample0, G, C, T, m, M, Mp, win, tw, spec, s2_auto, acc2, \
                n_s2, pref2, oi, lc, smem, stream, acc1, mode
  switch (oi.fmt) {
    case kImageGramTF32:
      return f32 ? launch_k1_t<SS_F32, kImageGramTF32>(K1_ARGS)
                 : launch_k1_t<SS_I16, kImageGramTF32>(K1_ARGS);
    case kImageGramBF16:
      return f32 ? launch_k1_t<SS_F32, kImageGramBF16>(K1_ARGS)
                 : launch_k1_t<SS_I16, kImageGramBF16>(K1_ARGS);
    case kImageGramF32:
      return f32 ? launch_k1_t<SS_F32, kImageGramF32>(K1_ARGS)
                 : launch_k1_t<SS_I16, kImageGramF32>(K1_ARGS);
    case kImageGramF16:
      return f32 ? launch_k1_t<SS_F32, kImageGramF16>(K1_ARGS)
                 : launch_k1_t<SS_I16, kImageGramF16>(K1_ARGS);
    default:
      return f32 ? launch_k1_t<SS_F32, kImageNone>(K1_ARGS)
                 : launch_k1_t<SS_I16, kImageNone>(K1_ARGS);
  }
#undef K1_ARGS
}

cudaError_t launch_k1_cross_s2(const float2* spec, long long chan_stride, int G, int m, int M,
                               int Mp, const int4* pairs, int n_pairs, float pref2, double* acc2,
                               long long plane, int nsm, cudaStream_t stream) {
  if (G <= 0 || n_pairs <= 0) return cudaSuccess;
  const int bx = (M + 127) / 128;
  int splits = std::max(1, (4 * nsm) / std::max(1, bx * n_pairs));
  splits = std::min(splits, std::max(1, G / 8));
  // at most kMaxFp32Groups groups in a thread's float32 sums (grid y <= 65535)
  splits = std::min(65535, std::max(splits, (G + kMaxFp32Groups - 1) / kMaxFp32Groups));
  const int gpc = (G + splits - 1) / splits;
  splits = (G + gpc - 1) / gpc;
  dim3 grid(bx, splits, n_pairs);
  k1_cross_s2<<<grid, 128, 0, stream>>>(spec, chan_stride, G, m, M, Mp, pairs, gpc, pref2, acc2,
                                        plane);
  return cudaGetLastError();
}

}  // namespace ss
