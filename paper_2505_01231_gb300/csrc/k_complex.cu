// k_complex.cu -- spectra of complex-valued signals (App. D) and S4 planes
// shifted off the cut (App. E), on CUDA cores (FP32, float64 across groups).
//
// A complex signal z = x + j y is carried as its two real channels, so K1's
// centred half spectra serve it: by the linearity of Eq. 18 and of the
// centring, the transform of z at a signed bin k is Z(k) = X(k) + j Y(k), with
// X(-k) = X(k)* for the real parts; the transform of z* at k is
// Z(-k)* = X(k) - j Y(k).  An operand is (real channel, imaginary channel or
// -1, conjugate flag): its value at k is X(k) + sigma j Y(k), sigma = +1 or -1.
// The k-statistics of Eq. 32-34 (App. H, Eq. 85 for the fourth order) are then
// taken directly over these complex samples -- the multilinear extension of
// Eq. 47, 48, 50 that App. D writes as sums of 4, 8 or 16 real spectra, formed
// here per group so that the error bars of Eq. 35-36 hold for the combination:
//   S2(k)    = c2(A(k), B(-k)),                      k in [-(M-1), M-1]
//   S3(k, l) = c3(A(k), B(l), C(-k-l)),              |k|, |l|, |k+l| <= M-1
//   S4(k, l) = c4(A(k+s), B(-k-s), C(l-s), D(-l+s)), |k|, |l| <= M-1
// (the window and dt normalisation is applied by K4).  s shifts the S4 plane
// of the 3-D trispectrum (App. E); bins are taken mod T (the transform of a
// frame is periodic in k).  Outputs: row r holds k = r - (M-1), column c holds
// l = c - (M-1).
//
// Bins repeat after T = 2 (M - 1), so row and column M - 1 repeat row and column
// -(M - 1): the kernels compute T x T points and store the first row and column
// twice.  (On the 2M - 1 = T + 1 rows and columns themselves the tiles of a power of
// two T were 1.7 times the plane's points at T = 128.)
//
// Bound by the FP32 ALUs: S4 takes 22 multiply-adds per point and frame, S3 8.  CTA =
// (tile, run of at most kMaxFp32Groups groups, combination), 128 threads.  The run's
// frames are one sequence, staged eight at a time with the same threads forming the
// same operands from frame to frame (bin, sign and addresses found once).  Points per
// thread so that shared memory, at 128 bytes a clock, keeps up with the multiply-adds:
// S4 2 x 4 (144 bytes for 176), S3 4 x 4 (128 bytes for 128).  A run's float32 sums go
// to the float64 accumulators.  One signal's S2, S3 and S4 over 2^19 samples (T = 128,
// m = 8; a pass with K1 and the results' copy): 583 us with one row x four columns a
// thread over the 2M - 1 rows and operands formed from scratch at every frame, 262 now.
#include <algorithm>

#include "internal.cuh"

namespace ss {
namespace {

constexpr int kThreads = 128, kChunk = 8;  // frames staged at a time
constexpr int kT4 = 32;                    // S4 tile: 32 x 32
constexpr int kR3 = 32, kL3 = 64;          // S3 tile
constexpr int kBins2 = 32, kLanes2 = 8;    // S2: bins of a CTA, its groups at a time

__device__ __forceinline__ float2 cmulc(float2 a, float2 b) {
  return make_float2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
}
__device__ __forceinline__ void cmacc(float2& acc, float2 a, float2 b) {
  acc.x = fmaf(a.x, b.x, fmaf(-a.y, b.y, acc.x));
  acc.y = fmaf(a.x, b.y, fmaf(a.y, b.x, acc.y));
}

// signed bin k wrapped into [-(T/2), T/2] (T = 2 (M - 1))
__device__ __forceinline__ int wrap_bin(int k, int M) {
  const int T = 2 * (M - 1);
  int r = (k + (M - 1)) % T;
  if (r < 0) r += T;
  return r - (M - 1);
}

// An operand (re channel, im channel or -1, sign of j) at one signed bin, to be read
// frame by frame: X(k) + sigma j Y(k) from the half spectra of the channels.
struct Operand {
  const float2* re;
  const float2* im;  // nullptr: a real signal
  float conj, sigma;

  __device__ __forceinline__ Operand(const float2* __restrict__ spec, long long chan_stride, int4 o,
                                     int k, int M) {
    k = wrap_bin(k, M);
    re = spec + o.x * chan_stride + abs(k);
    im = o.y >= 0 ? spec + o.y * chan_stride + abs(k) : nullptr;
    conj = k < 0 ? -1.f : 1.f;
    sigma = (float)o.z;
  }
  __device__ __forceinline__ float2 at(long long off) const {
    float2 v = re[off];
    v.y *= conj;
    if (im) {
      const float2 w = im[off];
      v.x -= sigma * (conj * w.y);
      v.y += sigma * w.x;
    }
    return v;
  }
};

__device__ __forceinline__ void flush4(double* __restrict__ acc, long long plane, long long o,
                                       float sr, float si, float qr, float qi) {
  atomicAdd(acc + o, widen(sr));
  atomicAdd(acc + plane + o, widen(si));
  atomicAdd(acc + 2 * plane + o, widen(qr));
  atomicAdd(acc + 3 * plane + o, widen(qi));
}

// S2: CTA = (32 bins, run of groups, combination); 8 groups at a time, their sums
// added in shared memory.  (One group a thread and four float64 additions for it took
// 19 us at T = 128, m = 8, 512 groups.)
__global__ void __launch_bounds__(kBins2 * kLanes2)
k5_cplx_s2(const float2* __restrict__ spec, long long chan_stride, int G, int m, int M, int Mp,
           const int4* __restrict__ ops, int groups_per_cta, float pref2,
           double* __restrict__ acc, long long plane) {
  __shared__ float4 part[kLanes2][kBins2];
  const int bin = threadIdx.x % kBins2, lane = threadIdx.x / kBins2;
  const int r = blockIdx.x * kBins2 + bin, n = 2 * M - 1;
  const int k = r - (M - 1);
  const Operand a(spec, chan_stride, ops[2 * blockIdx.z], k, M);
  const Operand b(spec, chan_stride, ops[2 * blockIdx.z + 1], -k, M);
  const int g0 = blockIdx.y * groups_per_cta, g1 = min(G, g0 + groups_per_cta);
  float sr = 0.f, si = 0.f, qr = 0.f, qi = 0.f;
  for (int g = g0 + lane; g < g1; g += kLanes2) {
    float2 c = make_float2(0.f, 0.f);
    long long off = (long long)g * m * Mp;
#pragma unroll 4
    for (int j = 0; j < m; ++j, off += Mp) cmacc(c, a.at(off), b.at(off));
    c.x *= pref2;
    c.y *= pref2;
    sr += c.x;
    si += c.y;
    qr = fmaf(c.x, c.x, qr);
    qi = fmaf(c.y, c.y, qi);
  }
  part[lane][bin] = make_float4(sr, si, qr, qi);
  __syncthreads();
  if (lane) return;
  for (int i = 1; i < kLanes2; ++i) {
    const float4 v = part[i][bin];
    sr += v.x;
    si += v.y;
    qr += v.z;
    qi += v.w;
  }
  if (r >= n - 1) return;
  const long long o = (long long)blockIdx.z * n;
  flush4(acc, plane, o + r, sr, si, qr, qi);
  if (r == 0) flush4(acc, plane, o + n - 1, sr, si, qr, qi);
}

// flush one point of the T x T plane to the places of the (2M - 1)^2 plane that it
// stands for, those within |k + l| <= kmax
__device__ __forceinline__ void flush_point(double* __restrict__ acc, long long plane, int n, int r,
                                            int c, int kmax, float sr, float si, float qr,
                                            float qi) {
  const int M1 = (n - 1) / 2;
  if (r >= n - 1 || c >= n - 1) return;
  for (int i = 0; i < (r == 0 ? 2 : 1); ++i)
    for (int j = 0; j < (c == 0 ? 2 : 1); ++j) {
      const int rr = i ? n - 1 : r, cc = j ? n - 1 : c;
      if (abs(rr + cc - 2 * M1) <= kmax)
        flush4(acc, plane, (long long)rr * n + cc, sr, si, qr, qi);
    }
}

// S3: thread = 4 x 4 points.  A frame's operands: a[32] | b[64] | c[96], c at
// -(k + l) for row + column = 0 .. 94; the 16-byte pieces of c are exchanged in pairs
// in every other 128 bytes, for the lanes of a row that lie 128 bytes apart.
__global__ void __launch_bounds__(kThreads, kRunCtas)
k5_cplx_s3(const float2* __restrict__ spec, long long chan_stride, int G, int m, int M, int Mp,
           const int4* __restrict__ ops, int tiles_l, int groups_per_cta, float pref3,
           double* __restrict__ acc, long long plane) {
  constexpr int kTasks = kR3 + kL3 + kR3 + kL3;
  __shared__ __align__(16) float2 st[kChunk][kTasks];
  const int tid = threadIdx.x;
  const int n = 2 * M - 1;
  const int r0 = (blockIdx.x / tiles_l) * kR3, c0 = (blockIdx.x % tiles_l) * kL3;
  const int g0 = blockIdx.y * groups_per_cta, g1 = min(G, g0 + groups_per_cta);
  if (g0 >= g1) return;
  const int kmin = r0 - (M - 1), lmin = c0 - (M - 1);
  // a tile off |k + l| <= M - 1 has nothing to compute, unless it holds a row or
  // column that stands for two
  if (r0 > 0 && c0 > 0 && (kmin + lmin > M - 1 || kmin + lmin + kR3 + kL3 - 2 < -(M - 1))) return;
  // operands formed by this thread: entries tid and 128 + tid (the latter: b[32 ..], c[64 ..])
  const int4 oa = ops[3 * blockIdx.z], ob = ops[3 * blockIdx.z + 1], oc = ops[3 * blockIdx.z + 2];
  const bool two = tid < kTasks - kThreads;
  const Operand op1(spec, chan_stride, tid < kR3 ? oa : tid < kR3 + kL3 ? ob : oc,
                    tid < kR3         ? kmin + tid
                    : tid < kR3 + kL3 ? lmin + tid - kR3
                                      : -(kmin + lmin + tid - kR3 - kL3),
                    M);
  const Operand op2(spec, chan_stride, oc, -(kmin + lmin + tid + kThreads - kR3 - kL3), M);
  // place of entry e (c exchanged)
  auto place = [](int e) {
    if (e < kR3 + kL3) return e;
    const int q = e - kR3 - kL3;
    return kR3 + kL3 + (q ^ (((q >> 4) & 1) << 1));
  };
  const int at1 = place(tid), at2 = place(tid + kThreads);
  // rows 4 ti .., columns 4 tj ..: a quarter warp reads 4 row sets, 2 column sets and
  // 5 diagonal sets
  const int lane = tid & 31, warp = tid >> 5;
  const int ti = (lane & 3) + 4 * (warp & 1), tj = (lane >> 2) + 8 * (warp >> 1);
  const int s0 = 4 * (ti + tj), s1 = s0 + 4;
  const int d0 = kR3 + kL3 + (s0 ^ (((s0 >> 4) & 1) << 1)), d1 = kR3 + kL3 + (s1 ^ (((s1 >> 4) & 1) << 1));
  float2 s[16];
  float sr[16], si[16], qr[16], qi[16];
#pragma unroll
  for (int p = 0; p < 16; ++p) {
    s[p] = make_float2(0.f, 0.f);
    sr[p] = si[p] = qr[p] = qi[p] = 0.f;
  }
  long long off = (long long)g0 * m * Mp;
  int j = 0;
  for (int left = (g1 - g0) * m; left > 0; left -= kChunk) {
    const int nf = min(kChunk, left);
    __syncthreads();  // the previous chunk has been read
#pragma unroll 4
    for (int f = 0; f < nf; ++f, off += Mp) {
      st[f][at1] = op1.at(off);
      if (two) st[f][at2] = op2.at(off);
    }
    __syncthreads();
#pragma unroll 1
    for (int f = 0; f < nf; ++f) {
      float2 a[4], b[4], c[8];
      const float2* row = st[f];
#pragma unroll
      for (int q = 0; q < 2; ++q) {
        const float4 u = reinterpret_cast<const float4*>(row + 4 * ti)[q];
        a[2 * q] = make_float2(u.x, u.y);
        a[2 * q + 1] = make_float2(u.z, u.w);
        const float4 v = reinterpret_cast<const float4*>(row + kR3 + 4 * tj)[q];
        b[2 * q] = make_float2(v.x, v.y);
        b[2 * q + 1] = make_float2(v.z, v.w);
        const float4 w = *reinterpret_cast<const float4*>(row + (d0 ^ (2 * q)));
        c[2 * q] = make_float2(w.x, w.y);
        c[2 * q + 1] = make_float2(w.z, w.w);
        const float4 z = *reinterpret_cast<const float4*>(row + (d1 ^ (2 * q)));
        c[4 + 2 * q] = make_float2(z.x, z.y);
        c[5 + 2 * q] = make_float2(z.z, z.w);
      }
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int h = 0; h < 4; ++h) cmacc(s[4 * i + h], cmulc(a[i], b[h]), c[i + h]);
      if (++j < m) continue;
      j = 0;
#pragma unroll
      for (int p = 0; p < 16; ++p) {
        const float cr = s[p].x * pref3, ci = s[p].y * pref3;
        sr[p] += cr;
        si[p] += ci;
        qr[p] = fmaf(cr, cr, qr[p]);
        qi[p] = fmaf(ci, ci, qi[p]);
        s[p] = make_float2(0.f, 0.f);
      }
    }
  }
  acc += (long long)blockIdx.z * n * n;
#pragma unroll
  for (int p = 0; p < 16; ++p)
    flush_point(acc, plane, n, r0 + 4 * ti + p / 4, c0 + 4 * tj + p % 4, M - 1, sr[p], si[p], qr[p],
                qi[p]);
}

// S4: thread = 2 x 4 points.  Thread e forms one operand of a frame: x = A(k + s) and
// y = B(-k - s) of row e / 2 < 32, z = C(l - s) and w = D(-l + s) of column e / 2 - 32, in
// even and odd threads; the even one also writes the product, and at a group's last frame
// the group's sum of it (the two sums that belong to a row or a column, not to a point).
__global__ void __launch_bounds__(kThreads, kRunCtas)
k5_cplx_s4(const float2* __restrict__ spec, long long chan_stride, int G, int m, int M, int Mp,
           const int4* __restrict__ ops, int tiles_l, int groups_per_cta, int shift, float pref,
           float fmm, float fm1, double* __restrict__ acc, long long plane) {
  // x or z, y or w, their product, the group's sum of the product; rows, then columns
  __shared__ __align__(16) float2 st[kChunk][4][2 * kT4];
  const int tid = threadIdx.x;
  const int n = 2 * M - 1;
  const int r0 = (blockIdx.x / tiles_l) * kT4, c0 = (blockIdx.x % tiles_l) * kT4;
  const int g0 = blockIdx.y * groups_per_cta, g1 = min(G, g0 + groups_per_cta);
  if (g0 >= g1) return;
  const int e = tid >> 1, odd = tid & 1, col = e >= kT4;
  const int bin = col ? c0 + e - kT4 - (M - 1) - shift : r0 + e - (M - 1) + shift;
  const Operand op(spec, chan_stride, ops[4 * blockIdx.z + 2 * col + odd], odd ? -bin : bin, M);
  const int lane = tid & 31, warp = tid >> 5;
  const int ti = (lane & 7) + 8 * (warp & 1), tj = (lane >> 3) + 4 * (warp >> 1);
  float2 a_xyzw[8], a_xz[8], a_yw[8], a_xw[8], a_yz[8];
  float sr[8], si[8], qr[8], qi[8];
#pragma unroll
  for (int p = 0; p < 8; ++p) {
    a_xyzw[p] = a_xz[p] = a_yw[p] = a_xw[p] = a_yz[p] = make_float2(0.f, 0.f);
    sr[p] = si[p] = qr[p] = qi[p] = 0.f;
  }
  float2 sum = make_float2(0.f, 0.f);  // even threads: the group's products so far
  long long off = (long long)g0 * m * Mp;
  int j = 0, js = 0;  // frame of the group: read, staged
  for (int left = (g1 - g0) * m; left > 0; left -= kChunk) {
    const int nf = min(kChunk, left);
    __syncthreads();  // the previous chunk has been read
#pragma unroll 4
    for (int f = 0; f < nf; ++f, off += Mp) {
      const float2 v = op.at(off);
      st[f][odd][e] = v;
      float2 w;
      w.x = __shfl_xor_sync(~0u, v.x, 1);
      w.y = __shfl_xor_sync(~0u, v.y, 1);
      const float2 vw = cmulc(v, w);
      sum.x += vw.x;
      sum.y += vw.y;
      if (!odd) st[f][2][e] = vw;
      if (++js == m) {
        if (!odd) st[f][3][e] = sum;
        sum = make_float2(0.f, 0.f);
        js = 0;
      }
    }
    __syncthreads();
#pragma unroll 1
    for (int f = 0; f < nf; ++f) {
      const float4 xv = reinterpret_cast<const float4*>(st[f][0])[ti];
      const float4 yv = reinterpret_cast<const float4*>(st[f][1])[ti];
      const float4 pv = reinterpret_cast<const float4*>(st[f][2])[ti];
      const float2 x[2] = {{xv.x, xv.y}, {xv.z, xv.w}}, y[2] = {{yv.x, yv.y}, {yv.z, yv.w}};
      const float2 xy[2] = {{pv.x, pv.y}, {pv.z, pv.w}};
#pragma unroll
      for (int q = 0; q < 2; ++q) {
        const int at = kT4 / 2 + 2 * tj + q;
        const float4 zv = reinterpret_cast<const float4*>(st[f][0])[at];
        const float4 wv = reinterpret_cast<const float4*>(st[f][1])[at];
        const float4 rv = reinterpret_cast<const float4*>(st[f][2])[at];
        const float2 z[2] = {{zv.x, zv.y}, {zv.z, zv.w}}, w[2] = {{wv.x, wv.y}, {wv.z, wv.w}};
        const float2 zw[2] = {{rv.x, rv.y}, {rv.z, rv.w}};
#pragma unroll
        for (int i = 0; i < 2; ++i)
#pragma unroll
          for (int h = 0; h < 2; ++h) {
            const int p = 4 * i + 2 * q + h;
            cmacc(a_xyzw[p], xy[i], zw[h]);
            cmacc(a_xz[p], x[i], z[h]);
            cmacc(a_yw[p], y[i], w[h]);
            cmacc(a_xw[p], x[i], w[h]);
            cmacc(a_yz[p], y[i], z[h]);
          }
      }
      if (++j < m) continue;
      j = 0;
      // c4 (App. H, Eq. 85 with complex samples) of the group at the thread's points
#pragma unroll
      for (int p = 0; p < 8; ++p) {
        float2 t = cmulc(st[f][3][2 * ti + p / 4], st[f][3][kT4 + 4 * tj + p % 4]);
        cmacc(t, a_xz[p], a_yw[p]);
        cmacc(t, a_xw[p], a_yz[p]);
        const float cr = pref * fmaf(fmm, a_xyzw[p].x, -fm1 * t.x);
        const float ci = pref * fmaf(fmm, a_xyzw[p].y, -fm1 * t.y);
        sr[p] += cr;
        si[p] += ci;
        qr[p] = fmaf(cr, cr, qr[p]);
        qi[p] = fmaf(ci, ci, qi[p]);
        a_xyzw[p] = a_xz[p] = a_yw[p] = a_xw[p] = a_yz[p] = make_float2(0.f, 0.f);
      }
    }
  }
  acc += (long long)blockIdx.z * n * n;
#pragma unroll
  for (int p = 0; p < 8; ++p)
    flush_point(acc, plane, n, r0 + 2 * ti + p / 4, c0 + 4 * tj + p % 4, 2 * M, sr[p], si[p], qr[p],
                qi[p]);
}

}  // namespace

cudaError_t launch_k5_complex(const float2* spec, long long chan_stride, int G, int m, int M,
                              int Mp, int order, const int4* ops, int n_combos, int shift,
                              bool natural, double* acc, long long plane, int nsm,
                              cudaStream_t stream) {
  if (G <= 0 || n_combos <= 0) return cudaSuccess;
  if (n_combos > 65535) return cudaErrorInvalidValue;
  const double md = m;
  const int n = 2 * M - 1;
  if (order == 2) {
    const int bx = (n - 1 + kBins2 - 1) / kBins2;
    const int runs = std::min((G + kLanes2 - 1) / kLanes2,
                              group_runs(G, (long long)bx * n_combos, nsm));
    const int gpc = (G + runs - 1) / runs;
    const float pref2 = (float)(natural ? 1.0 / md : 1.0 / (md - 1.0));
    k5_cplx_s2<<<dim3(bx, (G + gpc - 1) / gpc, n_combos), kBins2 * kLanes2, 0,
                 stream>>>(
        spec, chan_stride, G, m, M, Mp, ops, gpc, pref2, acc, plane);
    return cudaGetLastError();
  }
  const int th = order == 3 ? kR3 : kT4, tw = order == 3 ? kL3 : kT4;
  const int tiles_r = (n - 1 + th - 1) / th, tiles_l = (n - 1 + tw - 1) / tw;
  const long long tiles = (long long)tiles_r * tiles_l;
  if (tiles > 0x7fffffffll) return cudaErrorInvalidValue;
  const int runs = group_runs(G, tiles * n_combos, nsm);
  const int gpc = (G + runs - 1) / runs;
  const dim3 grid((unsigned)tiles, (unsigned)((G + gpc - 1) / gpc), (unsigned)n_combos);
  if (order == 3) {
    const float pref3 = (float)(natural ? 1.0 / md : md / ((md - 1.0) * (md - 2.0)));
    k5_cplx_s3<<<grid, kThreads, 0, stream>>>(spec, chan_stride, G, m, M, Mp, ops, tiles_l, gpc,
                                              pref3, acc, plane);
  } else {
    const float pref =
        (float)(natural ? 1.0 / (md * md) : 1.0 / ((md - 1.0) * (md - 2.0) * (md - 3.0)));
    const float fmm = (float)(natural ? md : md * (md + 1.0));
    const float fm1 = (float)(natural ? 1.0 : md - 1.0);
    k5_cplx_s4<<<grid, kThreads, 0, stream>>>(spec, chan_stride, G, m, M, Mp, ops, tiles_l, gpc,
                                              shift, pref, fmm, fm1, acc, plane);
  }
  return cudaGetLastError();
}

}  // namespace ss
