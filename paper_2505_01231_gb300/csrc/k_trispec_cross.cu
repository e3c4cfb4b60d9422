// k_trispec_cross.cu -- K3 for several channels: per-group trispectrum-cut
// k-statistics C4(a_k, b_k*, c_l, d_l*) (Sec. 7, Eq. 50) on CUDA cores (FP32).
//
// Domain: k in [-(M-1), M-1] (row r = k + M - 1 of the output grid), l in
// [0, M-1], with a_{-k} = a_k* (real channels).  With centred coefficients and,
// per group, x_j = da_jk, y_j = db_jk*, z_j = dc_jl, w_j = dd_jl*, the
// factorised estimator of App. H, Eq. 85 is
//   c4 = [m(m+1) sum xyzw - (m-1)(sum xy sum zw + sum xz sum yw + sum xw sum yz)]
//        / ((m-1)(m-2)(m-3)),
// all sums over the group's m frames and all products complex.  Per grid point
// and frame that is five complex multiply-adds (20 FFMA); sum xy and sum zw
// depend on one bin only.  The cut is complex for distinct channels, so the
// real and imaginary parts, their sums and their sums of squares over groups
// are accumulated (Eq. 35-36).
//
// Bound by the FP32 ALUs (22 operations a point and frame).  CTA = (32 x 32 tile of
// (r, l) of one combination, run of at most kMaxFp32Groups groups), 128 threads of 2 x 4
// points: 144 bytes of shared memory a frame for 176 operations, 32 lanes at 128 bytes a
// clock against 128 lanes of arithmetic.  The run's frames are one sequence, staged eight
// at a time; each thread forms the same operand from frame to frame.  Sums over groups
// stay in FP32 registers, then go to the float64 accumulators.  With M - 1 a multiple of
// 32 (T >= 64) the tiles leave out the last column and the mirrored combinations' last
// row, which k3_cross_last_col and k3_cross_last_row compute: of the (M - 1)/32 + 1 tiles
// a side would hold otherwise, the last held one line.  Six combinations of two channels,
// 2^20 samples, T = 256, m = 8: 1.19 ms with 1 x 4 points a thread and
// 16 x 64 tiles, 0.55 now.
#include "internal.cuh"

namespace ss {
namespace {

constexpr int kRT = kCrossRows32, kLT = kCrossRows32, kThreads = 128, kChunk = 8;

__device__ __forceinline__ float2 cmul(float2 a, float2 b) {
  return make_float2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
}
__device__ __forceinline__ void cmac(float2& acc, float2 a, float2 b) {
  acc.x = fmaf(a.x, b.x, fmaf(-a.y, b.y, acc.x));
  acc.y = fmaf(a.x, b.y, fmaf(a.y, b.x, acc.y));
}
__device__ __forceinline__ float2 conjf2(float2 a) { return make_float2(a.x, -a.y); }

__global__ void __launch_bounds__(kThreads, kRunCtas)
k3_trispec_cross(const float2* __restrict__ spec, long long chan_stride, int G, int m, int M,
                 int Mp, const int4* __restrict__ combos,
                 const int2* __restrict__ rowtiles, int tiles_l, int groups_per_cta,
                 float pref, float fmm, float fm1, double* __restrict__ acc, long long plane,
                 long long combo_stride) {
  // x or z, y or w, their product, the group's sum of the product; rows, then columns
  __shared__ __align__(16) float2 st[kChunk][4][kRT + kLT];
  const int tid = threadIdx.x;
  const int2 rt = rowtiles[blockIdx.x / tiles_l];  // (combination, first row)
  const int r0 = rt.y, l0 = (blockIdx.x % tiles_l) * kLT;
  const int g0 = blockIdx.y * groups_per_cta;
  const int g1 = min(G, g0 + groups_per_cta);
  if (g0 >= g1) return;
  const int rows = 2 * M - 1;
  // thread e / 2 of the rows, then of the columns; even: x = a_k or z = c_l, odd:
  // y = b_k* or w = d_l*.  Rows and columns past the grid repeat its last one (their
  // points are not stored).
  const int e = tid >> 1, odd = tid & 1;
  const int4 cb = combos[rt.x];
  const int chan = e < kRT ? (odd ? cb.y : cb.x) : (odd ? cb.w : cb.z);
  const int bin = e < kRT ? min(r0 + e, rows - 1) - (M - 1) : min(l0 + e - kRT, M - 1);
  const float conj = (bin < 0) != (odd != 0) ? -1.f : 1.f;
  const float2* src = spec + chan * chan_stride + abs(bin) + (long long)g0 * m * Mp;
  const int lane = tid & 31, warp = tid >> 5;
  const int ti = (lane & 7) + 8 * (warp & 1), tj = (lane >> 3) + 4 * (warp >> 1);
  float2 a_xyzw[8], a_xz[8], a_yw[8], a_xw[8], a_yz[8];
  float sre[8], sim[8], qre[8], qim[8];
#pragma unroll
  for (int p = 0; p < 8; ++p) {
    a_xyzw[p] = a_xz[p] = a_yw[p] = a_xw[p] = a_yz[p] = make_float2(0.f, 0.f);
    sre[p] = sim[p] = qre[p] = qim[p] = 0.f;
  }
  float2 sum = make_float2(0.f, 0.f);  // even threads: the group's products so far
  int j = 0, js = 0;                   // frame of the group: read, staged
  for (int left = (g1 - g0) * m; left > 0; left -= kChunk) {
    const int nf = min(kChunk, left);
    __syncthreads();  // the previous chunk has been read
#pragma unroll 4
    for (int f = 0; f < nf; ++f, src += Mp) {
      float2 v = *src, w;
      v.y *= conj;
      st[f][odd][e] = v;
      w.x = __shfl_xor_sync(~0u, v.x, 1);
      w.y = __shfl_xor_sync(~0u, v.y, 1);
      const float2 vw = cmul(v, w);
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
        const int at = kRT / 2 + 2 * tj + q;
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
            cmac(a_xyzw[p], xy[i], zw[h]);
            cmac(a_xz[p], x[i], z[h]);
            cmac(a_yw[p], y[i], w[h]);
            cmac(a_xw[p], x[i], w[h]);
            cmac(a_yz[p], y[i], z[h]);
          }
      }
      if (++j < m) continue;
      j = 0;
      // c4 of this group at the thread's points
#pragma unroll
      for (int p = 0; p < 8; ++p) {
        float2 t = cmul(st[f][3][2 * ti + p / 4], st[f][3][kRT + 4 * tj + p % 4]);
        cmac(t, a_xz[p], a_yw[p]);
        cmac(t, a_xw[p], a_yz[p]);
        const float cr = pref * fmaf(fmm, a_xyzw[p].x, -fm1 * t.x);
        const float ci = pref * fmaf(fmm, a_xyzw[p].y, -fm1 * t.y);
        sre[p] += cr;
        sim[p] += ci;
        qre[p] = fmaf(cr, cr, qre[p]);
        qim[p] = fmaf(ci, ci, qim[p]);
        a_xyzw[p] = a_xz[p] = a_yw[p] = a_xw[p] = a_yz[p] = make_float2(0.f, 0.f);
      }
    }
  }
#pragma unroll
  for (int p = 0; p < 8; ++p) {
    const int r = r0 + 2 * ti + p / 4, l = l0 + 4 * tj + p % 4;
    if (r >= rows || l >= M) continue;
    const long long o = (long long)rt.x * combo_stride + (long long)r * M + l;
    atomicAdd(acc + o, widen(sre[p]));
    atomicAdd(acc + plane + o, widen(sim[p]));
    atomicAdd(acc + 2 * plane + o, widen(qre[p]));
    atomicAdd(acc + 3 * plane + o, widen(qim[p]));
  }
}

// One grid point (r, l) of a combination over the groups g0, g0 + step, ..., straight
// from memory, for the lines that the tiles leave out.
__device__ __forceinline__ void cross_point(const float2* __restrict__ spec, long long chan_stride,
                                            int G, int m, int M, int Mp, int4 cb, int r, int l,
                                            int g0, int step, float pref, float fmm, float fm1,
                                            double* __restrict__ acc, long long plane) {
  const int k = r - (M - 1);
  const float conj = k < 0 ? -1.f : 1.f;
  float sr = 0.f, si = 0.f, qr = 0.f, qi = 0.f;
  for (int g = g0; g < G; g += step) {
    const long long base = (long long)g * m * Mp;
    const float2* A = spec + cb.x * chan_stride + base + abs(k);
    const float2* B = spec + cb.y * chan_stride + base + abs(k);
    const float2* C = spec + cb.z * chan_stride + base + l;
    const float2* D = spec + cb.w * chan_stride + base + l;
    const float2 o = make_float2(0.f, 0.f);
    float2 xyzw = o, xz = o, yw = o, xw = o, yz = o, sxy = o, szw = o;
#pragma unroll 4
    for (int j = 0; j < m; ++j) {
      float2 x = __ldg(A + (long long)j * Mp), y = __ldg(B + (long long)j * Mp);
      const float2 z = __ldg(C + (long long)j * Mp), w = conjf2(__ldg(D + (long long)j * Mp));
      x.y *= conj;
      y.y *= -conj;
      const float2 xy = cmul(x, y), zw = cmul(z, w);
      cmac(xyzw, xy, zw);
      cmac(xz, x, z);
      cmac(yw, y, w);
      cmac(xw, x, w);
      cmac(yz, y, z);
      sxy = make_float2(sxy.x + xy.x, sxy.y + xy.y);
      szw = make_float2(szw.x + zw.x, szw.y + zw.y);
    }
    float2 t = cmul(sxy, szw);
    cmac(t, xz, yw);
    cmac(t, xw, yz);
    const float cr = pref * fmaf(fmm, xyzw.x, -fm1 * t.x);
    const float ci = pref * fmaf(fmm, xyzw.y, -fm1 * t.y);
    sr += cr;
    si += ci;
    qr = fmaf(cr, cr, qr);
    qi = fmaf(ci, ci, qi);
  }
  acc += (long long)r * M + l;
  atomicAdd(acc, widen(sr));
  atomicAdd(acc + plane, widen(si));
  atomicAdd(acc + 2 * plane, widen(qr));
  atomicAdd(acc + 3 * plane, widen(qi));
}

// The row k = M - 1 of the mirrored combinations (the tiles leave it out when it would be
// alone in one): thread = column, one group at a time.
constexpr int kRowThreads = 128;

__global__ void __launch_bounds__(kRowThreads)
k3_cross_last_row(const float2* __restrict__ spec, long long chan_stride, int G, int m, int M, int Mp,
                  const int4* __restrict__ combos, const int2* __restrict__ half, float pref,
                  float fmm, float fm1, double* __restrict__ acc, long long plane,
                  long long combo_stride) {
  const int l = blockIdx.x * kRowThreads + threadIdx.x, q = half[blockIdx.z].x;
  if (l >= M) return;
  cross_point(spec, chan_stride, G, m, M, Mp, combos[q], 2 * M - 2, l, blockIdx.y, gridDim.y, pref,
              fmm, fm1, acc + q * combo_stride, plane);
}

// The column l = M - 1 of the row tiles' rows: CTA = four row tiles, warp = one, thread =
// row, one group at a time.
__global__ void __launch_bounds__(4 * kRT)
k3_cross_last_col(const float2* __restrict__ spec, long long chan_stride, int G, int m, int M, int Mp,
                  const int4* __restrict__ combos, const int2* __restrict__ rowtiles, int n_rowtiles,
                  float pref, float fmm, float fm1, double* __restrict__ acc, long long plane,
                  long long combo_stride) {
  const int i = 4 * blockIdx.x + threadIdx.x / kRT;
  if (i >= n_rowtiles) return;
  const int2 rt = rowtiles[i];
  const int r = rt.y + threadIdx.x % kRT;
  if (r >= 2 * M - 1) return;
  cross_point(spec, chan_stride, G, m, M, Mp, combos[rt.x], r, M - 1, blockIdx.y, gridDim.y, pref,
              fmm, fm1, acc + rt.x * combo_stride, plane);
}

// blockIdx.z: combination (of the mirrored ones) x plane; rows r < M - 1 from 2M - 2 - r
__global__ void k3_cross_mirror(double* __restrict__ acc, const int2* __restrict__ half, int M,
                                long long combo_stride, long long plane) {
  const int2 h = half[blockIdx.z >> 2];
  const int pl = blockIdx.z & 3;
  double* a = acc + pl * plane + h.x * combo_stride;
  const bool negate = h.y != 0 && pl == 1;  // the sum of Im of the conjugate
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < (M - 1) * M; i += gridDim.x * blockDim.x) {
    const int r = i / M, l = i - r * M;
    const double v = a[(long long)(2 * M - 2 - r) * M + l];
    a[i] = negate ? __hiloint2double(__double2hiint(v) ^ 0x80000000, __double2loint(v)) : v;
  }
}

// row r = 0 (k = -(M - 1)) of every plane and combination <- row r = 2M - 2
__global__ void k3_cross_row0(double* __restrict__ acc, int n, int M, long long combo_stride,
                              long long plane) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const int l = i % M, pc = i / M;
  const int c = pc >> 2, pl = pc & 3;
  double* a = acc + pl * plane + (long long)c * combo_stride;
  a[l] = a[(long long)(2 * M - 2) * M + l];
}

// Runs of groups of the kernels of single lines: some 4096 CTAs, but four groups a thread
// where they last (each thread adds its sums in float64 to the same places) and at most
// kMaxFp32Groups.
int edge_runs(int G, int ctas_per_run) {
  int runs = std::min((G + 3) / 4, std::max(1, 4096 / ctas_per_run));
  runs = std::max(runs, (G + kMaxFp32Groups - 1) / kMaxFp32Groups);
  return std::min(runs, 65535);
}

}  // namespace

cudaError_t launch_k3_cross_last_row(const float2* spec, long long chan_stride, int G, int m, int M,
                                     int Mp, const int4* combos, const CrossTiles& ct, float pref,
                                     float fmm, float fm1, double* acc, long long plane,
                                     cudaStream_t stream) {
  if (ct.n_half <= 0) return cudaSuccess;
  const int gx = (M + kRowThreads - 1) / kRowThreads;
  const int gy = edge_runs(G, gx * ct.n_half);
  k3_cross_last_row<<<dim3((unsigned)gx, (unsigned)gy, (unsigned)ct.n_half), kRowThreads, 0, stream>>>(
      spec, chan_stride, G, m, M, Mp, combos, ct.half, pref, fmm, fm1, acc, plane,
      (long long)(2 * M - 1) * M);
  return cudaGetLastError();
}

cudaError_t launch_k3_cross_mirror(const CrossTiles& ct, int n_combos, int M, double* acc,
                                   long long plane, bool row0, cudaStream_t stream) {
  const long long combo_stride = (long long)(2 * M - 1) * M;
  if (row0) {
    const int n = 4 * n_combos * M;
    k3_cross_row0<<<(n + 255) / 256, 256, 0, stream>>>(acc, n, M, combo_stride, plane);
    const cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
  }
  if (ct.n_half > 0) {
    const int gx = std::min(256, ((M - 1) * M + 255) / 256);
    k3_cross_mirror<<<dim3((unsigned)gx, 1, (unsigned)(4 * ct.n_half)), 256, 0, stream>>>(
        acc, ct.half, M, combo_stride, plane);
  }
  return cudaGetLastError();
}

cudaError_t launch_k3_trispec_cross(const float2* spec, long long chan_stride, int G, int m, int M,
                                    int Mp, const int4* combos, int n_combos, const CrossTiles& ct,
                                    double* acc, long long plane, int nsm, bool natural,
                                    cudaStream_t stream) {
  if (G <= 0 || n_combos <= 0) return cudaSuccess;
  const int rows = 2 * M - 1;
  const bool edges = (M - 1) % kCrossRows32 == 0;
  const int tiles_l = edges ? (M - 1) / kLT : (M + kLT - 1) / kLT;
  const long long tiles = (long long)ct.n_rowtiles * tiles_l;  // of all combinations
  if (tiles > 0x7fffffffll || 4 * ct.n_half > 65535) return cudaErrorInvalidValue;
  const int runs = group_runs(G, tiles, nsm);
  const int gpc = (G + runs - 1) / runs;
  const double md = m;
  // c4 = pref [fmm sum xyzw - fm1 (sum xy sum zw + ...)]: the k-statistic (Eq. 85),
  // or the natural estimator 1/m sum xyzw - 1/m^2 (...)
  const float pref =
      (float)(natural ? 1.0 / (md * md) : 1.0 / ((md - 1.0) * (md - 2.0) * (md - 3.0)));
  const float fmm = (float)(natural ? md : md * (md + 1.0));
  const float fm1 = (float)(natural ? 1.0 : md - 1.0);
  const dim3 grid((unsigned)tiles, (unsigned)((G + gpc - 1) / gpc));
  const long long combo_stride = (long long)rows * M;
  k3_trispec_cross<<<grid, kThreads, 0, stream>>>(spec, chan_stride, G, m, M, Mp, combos, ct.rowtiles,
                                                  tiles_l, gpc, pref, fmm, fm1, acc, plane,
                                                  combo_stride);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  if (edges) {
    const int gx = (ct.n_rowtiles + 3) / 4;
    const int gy = edge_runs(G, gx);
    k3_cross_last_col<<<dim3((unsigned)gx, (unsigned)gy), 4 * kRT, 0, stream>>>(
        spec, chan_stride, G, m, M, Mp, combos, ct.rowtiles, ct.n_rowtiles, pref, fmm, fm1, acc,
        plane, combo_stride);
    e = cudaGetLastError();
    if (e == cudaSuccess)
      e = launch_k3_cross_last_row(spec, chan_stride, G, m, M, Mp, combos, ct, pref, fmm, fm1, acc,
                                   plane, stream);
    if (e != cudaSuccess) return e;
  }
  return launch_k3_cross_mirror(ct, n_combos, M, acc, plane, true, stream);
}

}  // namespace ss
