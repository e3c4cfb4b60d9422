// k_finalize.cu -- K4: mean over groups and standard errors, in float64; and the
// element-wise float64 addition that merges the group sums of two plans.
//
// For every output grid point it reads the float64 sums over the G groups of
// S_g (real and imaginary part) and of their squares, applies the window and
// dt normalisation `norm` of Eq. 23, 28, 31 (and Eq. 47, 48, 50), and writes
//   mean = norm sum / G
//   err  = sqrt( G/(G-1) (norm^2 sumsq / G - mean^2) / G )   (Eq. 35-36)
// for the real and the imaginary part.  One-channel grids that were computed
// on the k <= l half are mirrored with S(k, l) = S(l, k) (Sec. 9), whether the
// sums of (k, l) are stored at [k][l] or at [l][k]; bispectrum points with
// k + l > M-1 are set to zero.
//
// One launch takes all orders of a plan (up to kK4Jobs grids).  It moves 32 bytes in (16
// for the real one-channel S4) and 32 out a point, but float64 bounds it: two operations a
// clock and SM, so the constants are the host's and the square root is k4_sqrt (four
// channels, T = 512: 85 grids of 132 000 points in 0.51 ms, with two divisions a
// point and sqrt 0.67 ms).  A mirrored grid goes in
// tiles of 32 x 32 points of the stored half, each read once in rows and written twice,
// as it is and transposed through shared memory: thread = output element instead read the
// mirrored half down the columns (T = 4096: 179 + 299 us for S3 and S4, now 123 us for
// both; T = 2048: 70 + 99 us, now 41 us).
#include <algorithm>

#include "internal.cuh"

namespace ss {
namespace {

constexpr int kK4Threads = 256, kK4Tile = 32, kK4PerThread = 4;

struct K4Value {
  double2 mean, err;
};

// sqrt(x) (0 for x <= 0) from the float32 reciprocal square root and two Newton steps
// r += (x - r^2) y / 2 in float64: 7 operations of the slow float64 pipe.  The float32
// start has a relative error of a few 1e-8 and so do the steps' factors y, so the first
// step leaves about 1e-14 and the second the rounding.  Values near the ends of the
// float32 range take sqrt itself.
__device__ __forceinline__ double k4_sqrt(double x) {
  const int e = (__double2hiint(x) >> 20) - 1023;  // negative x: below every exponent
  if (e > -100 && e < 100) {
    const double y = (double)rsqrtf((float)x), h = 0.5 * y;
    double r = x * y;
    r = fma(fma(-r, r, x), h, r);
    return fma(fma(-r, r, x), h, r);
  }
  return x > 0.0 ? sqrt(x) : 0.0;
}

__device__ __forceinline__ K4Value k4_value(const K4Job& j, const double* acc, const double* prev,
                                            long long o, bool real) {
  // the sums of the groups since the snapshot `prev` (a block of sequential spectra),
  // or of all groups
  auto sum = [&](int q) {
    const double s = acc[q * j.plane + o];
    return prev ? s - prev[q * j.plane + o] : s;
  };
  auto part = [&](int q, double* mean, double* err) {
    const double m = j.mean_scale * sum(q);
    *mean = m;
    *err = k4_sqrt(fma(j.sq_scale, sum(q + 2), -j.mean_sq_scale * (m * m)));
  };
  K4Value v{make_double2(0.0, 0.0), make_double2(0.0, 0.0)};
  part(0, &v.mean.x, &v.err.x);
  if (!real) part(1, &v.mean.y, &v.err.y);
  return v;
}

__global__ void __launch_bounds__(kK4Threads) k4_finalize(const __grid_constant__ K4Jobs js) {
  __shared__ double2 sm[kK4Tile][kK4Tile + 1], se[kK4Tile][kK4Tile + 1];
  int b = blockIdx.x, i = 0;
  while (i + 1 < js.n && b >= js.job[i + 1].first_block) ++i;
  const K4Job& j = js.job[i];
  b -= j.first_block;
  const double* acc = j.acc + blockIdx.y * j.acc_stride;
  const double* prev = j.prev;
  double* out = j.out ? j.out + blockIdx.y * j.out_stride : nullptr;
  double* err = j.err ? j.err + blockIdx.y * j.out_stride : nullptr;
  auto put = [&](long long e, const double2& m, const double2& s) {
    if (j.wide) {  // both 16-byte aligned
      if (out) *reinterpret_cast<double2*>(out + 2 * e) = m;
      if (err) *reinterpret_cast<double2*>(err + 2 * e) = s;
    } else {
      if (out) { out[2 * e] = m.x; out[2 * e + 1] = m.y; }
      if (err) { err[2 * e] = s.x; err[2 * e + 1] = s.y; }
    }
  };
  if (j.layout == kLayoutVector || j.layout == kLayoutCross) {
    const long long total = (long long)j.n_combos * j.rows * j.M;
#pragma unroll
    for (int q = 0; q < kK4PerThread; ++q) {
      const long long e = ((long long)b * kK4PerThread + q) * kK4Threads + threadIdx.x;
      if (e < total) {
        const K4Value v = k4_value(j, acc, prev, e, false);
        put(e, v.mean, v.err);
      }
    }
    return;
  }
  // tile pair (ta, tb), ta <= tb, of the triangle k <= l
  const int M = j.M, nt = (M + kK4Tile - 1) / kK4Tile, pairs = nt * (nt + 1) / 2;
  const int combo = b / pairs, t = b - combo * pairs;
  int tb = (int)((sqrtf(8.f * (float)t + 1.f) - 1.f) * 0.5f);
  while (tb * (tb + 1) / 2 > t) --tb;
  while ((tb + 1) * (tb + 2) / 2 <= t) ++tb;
  const int ta = t - tb * (tb + 1) / 2;
  const int k0 = ta * kK4Tile, l0 = tb * kK4Tile;
  const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
  const bool lower = j.layout == kLayoutS4Lower;  // (k, l) is stored at [l][k]
  const bool real = j.layout != kLayoutS3Single;
  const long long base = (long long)combo * M * M;
  // sm[r][c]: stored row r, column c of the tile
  for (int r = ty; r < kK4Tile; r += kK4Threads / 32) {
    const int k = k0 + (lower ? tx : r), l = l0 + (lower ? r : tx);
    K4Value v{make_double2(0.0, 0.0), make_double2(0.0, 0.0)};
    if (k <= l && l < M && (j.layout != kLayoutS3Single || k + l <= M - 1))
      v = k4_value(j, acc, prev, base + (lower ? (long long)l * M + k : (long long)k * M + l), real);
    sm[r][tx] = v.mean;
    se[r][tx] = v.err;
  }
  __syncthreads();
  // the point (k0 + a, l0 + c) of the tile
  auto point = [&](int a, int c, double2* m, double2* s) {
    *m = lower ? sm[c][a] : sm[a][c];
    *s = lower ? se[c][a] : se[a][c];
  };
  for (int r = ty; r < kK4Tile; r += kK4Threads / 32) {
    double2 m, s;
    if (k0 + r < M && l0 + tx < M) {  // output row k0 + r, column l0 + tx
      if (ta == tb && tx < r)
        point(tx, r, &m, &s);
      else
        point(r, tx, &m, &s);
      put(base + (long long)(k0 + r) * M + l0 + tx, m, s);
    }
    if (ta != tb && l0 + r < M && k0 + tx < M) {  // and its mirror image
      point(tx, r, &m, &s);
      put(base + (long long)(l0 + r) * M + k0 + tx, m, s);
    }
  }
}

__global__ void k_add_f64(double* __restrict__ dst, const double* __restrict__ src, long long n) {
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n;
       i += (long long)gridDim.x * blockDim.x)
    dst[i] += src[i];
}

__global__ void k_add_blocks(double* __restrict__ acc, double* __restrict__ prev,
                             const double* __restrict__ blk, long long stride, int n_blocks,
                             long long n) {
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n;
       i += (long long)gridDim.x * blockDim.x) {
    double s = acc[i];
#pragma unroll 8
    for (int b = 0; b < n_blocks; ++b) s += blk[b * stride + i];
    acc[i] = s;
    prev[i] = s;
  }
}

}  // namespace

cudaError_t launch_add_blocks(double* acc, double* prev, const double* blk, long long stride,
                              int n_blocks, long long n, cudaStream_t stream) {
  if (n <= 0) return cudaSuccess;
  const long long grid = std::min<long long>((n + 255) / 256, 4096);
  k_add_blocks<<<(int)grid, 256, 0, stream>>>(acc, prev, blk, stride, n_blocks, n);
  return cudaGetLastError();
}

cudaError_t launch_add_f64(double* dst, const double* src, long long n, cudaStream_t stream) {
  if (n <= 0) return cudaSuccess;
  long long grid = (n + 255) / 256;
  if (grid > 4096) grid = 4096;
  k_add_f64<<<(int)grid, 256, 0, stream>>>(dst, src, n);
  return cudaGetLastError();
}

K4Job k4_job(const double* acc, int n_combos, int rows, int M, int layout, long long G, double norm,
             double* out, double* err, const double* prev) {
  K4Job j{};
  j.acc = acc;
  j.prev = prev;
  j.out = out;
  j.err = err;
  j.plane = (long long)n_combos * rows * M;
  j.n_combos = n_combos;
  j.rows = rows;
  j.M = M;
  j.layout = layout;
  // mean = norm sum / G, err^2 = (norm^2 sumsq / G - mean^2) / (G - 1)
  const double g = (double)G;
  j.mean_scale = norm / g;
  j.sq_scale = norm * norm / (g * (g - 1.0));
  j.mean_sq_scale = 1.0 / (g - 1.0);
  return j;
}

cudaError_t launch_k4(K4Jobs& js, int n_blocks, cudaStream_t stream) {
  long long blocks = 0;
  int n = 0;
  for (int i = 0; i < js.n; ++i) {
    K4Job j = js.job[i];
    const long long total = (long long)j.n_combos * j.rows * j.M;
    if (total == 0 || (!j.out && !j.err)) continue;
    j.wide = (((uintptr_t)j.out | (uintptr_t)j.err) & 15) == 0 && (j.out_stride & 1) == 0;
    j.first_block = (int)blocks;
    const long long nt = (j.M + kK4Tile - 1) / kK4Tile;
    blocks += j.layout == kLayoutVector || j.layout == kLayoutCross
                  ? (total + kK4Threads * kK4PerThread - 1) / (kK4Threads * kK4PerThread)
                  : j.n_combos * (nt * (nt + 1) / 2);
    js.job[n++] = j;
  }
  js.n = n;
  if (n == 0 || n_blocks <= 0) return cudaSuccess;
  if (blocks > 0x7fffffffll) return cudaErrorInvalidValue;
  for (int y = 0; y < n_blocks; y += 65535) {
    K4Jobs part = js;
    for (int i = 0; i < n; ++i) {
      part.job[i].acc += y * part.job[i].acc_stride;
      if (part.job[i].out) part.job[i].out += y * part.job[i].out_stride;
      if (part.job[i].err) part.job[i].err += y * part.job[i].out_stride;
    }
    k4_finalize<<<dim3((unsigned)blocks, (unsigned)std::min(65535, n_blocks - y)), kK4Threads, 0,
                  stream>>>(part);
    const cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

cudaError_t launch_k4_finalize(const double* acc, int n_combos, int rows, int M, int layout,
                               long long G, double norm, double* out, double* err,
                               cudaStream_t stream, const double* prev) {
  K4Jobs js{};
  js.n = 1;
  js.job[0] = k4_job(acc, n_combos, rows, M, layout, G, norm, out, err, prev);
  return launch_k4(js, 1, stream);
}

}  // namespace ss
