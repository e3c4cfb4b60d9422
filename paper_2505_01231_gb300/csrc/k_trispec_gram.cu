// k_trispec_gram.cu -- K3 in FP32 on CUDA cores for small groups: the trispectrum
// cut (Eq. 31) with the factorised fourth k-statistic (App. H, Eq. 85) as one
// weighted contraction of the frame Gram per group.
//
// The bracket of Eq. 85 for (a_k, a_k*, a_l, a_l*) is sum_{j<=j'} w_jj' G^k_jj' G^l_jj'
// over the frame Gram G^k_jj' = Re(d_jk d_j'k*) of each bin (the algebra stands with
// OperandImage in internal.cuh), so c4 is one real dot product of K = m(m+1)/2 + 1
// entries per grid point and group.  K1 writes the entries of every bin in float32,
// one row of bins per entry: first the entries with negative weight (the pairs j < j'
// and ps), then the diagonal, then zero rows up to a multiple of 8.
//
// Against the five length-m sums per point of k3_trispec this is 58 instead of 62 FP
// operations a point and group at m = 10, but one accumulator a point instead of
// five: a thread holds 8 x 8 points (64 registers; their sums and sums of squares over
// the item's groups live in TMEM), so an entry costs 4 shared-memory loads of 16
// bytes per 64 FMAs instead of 6 per 80, with addresses that are constants of the
// unrolled loop, and 16 warps stay resident per SM instead of 8.  The FMAs go two to an
// instruction (fma.rn.f32x2 over neighbouring l): the FMA pipe does the same work, but
// half the issue slots are left for the loads and the pairs (a, a), and a packed
// operand reads both register banks at once.  The negative entries come first and the
// sums change sign once where they end, since a packed FMA cannot negate an operand.
// Measured, 2^25 samples, T = 1024, m = 10 (S4 with the column kernel): k3_trispec 2.11
// ms; this kernel with scalar FMAs 1.27 ms (FMA pipe 58 %, issue 75 %), with 8 x 16
// points a thread and 8 warps 1.51 ms, with packed FMAs 1.10 ms (FMA pipe 70 %, issue
// 57 %); K1 pays 0.05 ms for the operand image.  T = 512, m = 16, 2^23 samples: 0.30 ms.
// K grows as m^2, the five sums as m: the plan takes this form up to m = kGram32MaxM.
// The error against float64 is smaller too: 1.3e-7 of the norm instead of 4.2e-7.
//
// Work split as in k2_bispec84w: a 128-thread CTA takes (group chunk, 32 x 64 tile)
// items, each of its four warps a quarter of the item's groups; a warp stages 8 entry
// rows of its tile at a time (32 bins at k0, 64 at l0, two 2-D TMA boxes without
// swizzling) into its own ring.  Lane (tx, ty) = (lane & 3, lane >> 2) takes the k
// rows 4 tx + 0..3 and 16 + 4 tx + 0..3 and the l columns 4 ty + 0..3 and 32 + 4 ty +
// 0..3, so a warp's load of each operand is 64 or 128 consecutive bytes.  Every wait is
// bounded; a failure stops the CTA after its copies have landed.
#include <algorithm>

#include "internal.cuh"
#include "pipeline.cuh"

namespace ss {
namespace {

constexpr int kGThreads = 128, kGWarps = kGThreads / 32;
constexpr int kGRows = kGram32Rows;  // entry rows of a stage
constexpr int kGSt = 4;              // stages of a warp's ring
constexpr uint32_t kGA = kGRows * 32 * 4, kGB = kGRows * 64 * 4;
constexpr uint32_t kGStage = kGA + kGB;
constexpr uint32_t kGRing = kGSt * kGStage;  // 12 KB
constexpr uint32_t kGTmemCols = 128;         // 64 sums and 64 sums of squares a lane
static_assert(kGRing >= 32 * 64 * sizeof(float), "the flush exchanges one part in the ring");

__device__ __forceinline__ float4 lds128_g(uint32_t a) {
  float4 v;
  asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];"
               : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w)
               : "r"(a));
  return v;
}

__device__ __forceinline__ void tmem_ld16_g(uint32_t taddr, uint32_t (&r)[16]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,"
      "%14,%15}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
        "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]),
        "=r"(r[14]), "=r"(r[15])
      : "r"(taddr));
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
}

__device__ __forceinline__ void tmem_st16_g(uint32_t taddr, const uint32_t (&r)[16]) {
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,"
      "%13,%14,%15,%16};" ::"r"(taddr),
      "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]),
      "r"(r[8]), "r"(r[9]), "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15])
      : "memory");
}

__device__ __forceinline__ void tmem_wait_st_g() {
  asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
}

typedef unsigned long long f32x2;  // two floats, the first in the low half

__device__ __forceinline__ f32x2 pack2(float lo, float hi) {
  f32x2 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
  return r;
}
__device__ __forceinline__ float2 unpack2(f32x2 v) {
  float2 r;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(v));
  return r;
}
__device__ __forceinline__ void fma2(f32x2& acc, f32x2 a, f32x2 b) {
  asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(acc) : "l"(a), "l"(b));
}

// one entry row: acc[4 i + j] += (a_i, a_i) (b_2j, b_2j+1)
__device__ __forceinline__ void entry_row(uint32_t pa, uint32_t pb, f32x2 (&acc)[32]) {
  const float4 a0 = lds128_g(pa), a1 = lds128_g(pa + 64);
  const float a[8] = {a0.x, a0.y, a0.z, a0.w, a1.x, a1.y, a1.z, a1.w};
  f32x2 b[4];
#pragma unroll
  for (int h = 0; h < 2; ++h)
    asm volatile("ld.shared.v2.b64 {%0, %1}, [%2];"
                 : "=l"(b[2 * h]), "=l"(b[2 * h + 1])
                 : "r"(pb + 128 * h));
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const f32x2 aa = pack2(a[i], a[i]);
#pragma unroll
    for (int j = 0; j < 4; ++j) fma2(acc[4 * i + j], aa, b[j]);
  }
}

struct ItemGram {
  int k0, l0, row;    // tile, first entry row of the warp's groups
  long long acc_off;  // of the tile's row k0, column l0
};

__global__ void __launch_bounds__(kGThreads, 4)
k3_trispec_gram(const __grid_constant__ CUtensorMap tm32, const __grid_constant__ CUtensorMap tm64,
                int stages_per_group, int n_neg, int G, int M, int lim,
                const TileInfo* __restrict__ tiles, WarpQueue wq, double* __restrict__ acc,
                long long plane, int* __restrict__ status) {
  extern __shared__ __align__(1024) unsigned char smem_raw[];  // + 1024 spare bytes
  __shared__ __align__(8) uint64_t full[kGWarps][kGSt];
  __shared__ uint32_t tmem_slot;
  __shared__ ItemGram items[kGWarps];
  __shared__ int s_next;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  ItemGram& it = items[warp];
  unsigned char* ring0 = align1024<unsigned char>(smem_raw);
  unsigned char* ring = ring0 + (size_t)warp * kGRing;
  const int tx = lane & 3, ty = lane >> 2;
  const uint32_t ring_s = smem_addr(ring);

  if (tid == 0) {
    for (int w = 0; w < kGWarps; ++w)
      for (int s = 0; s < kGSt; ++s) mbar_init(&full[w][s], 1);
    fence_mbar_init();
  }
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                     smem_addr(&tmem_slot)),
                 "r"(kGTmemCols));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  fence_async_smem();
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tsum = tmem_slot + ((uint32_t)(32 * warp) << 16);
  uint32_t qb = 0;  // stages this warp has consumed (stage = q % kGSt)
  int next = 0;     // thread 0: the item after the current one, drawn while it runs
  if (tid == 0) next = draw_item(wq);
  for (;;) {
    if (tid == 0) s_next = next;
    __syncthreads();
    const int item = s_next;
    if (item >= wq.n_items) break;
    if (tid == 0) next = draw_item(wq);
    int nst;  // stages of the warp's groups, consecutive entry rows
    {
      const int chunk = item / wq.n_tiles, t = item - chunk * wq.n_tiles;
      const int blk = chunk / wq.chunks_per_block;
      int ga = blk * wq.block_groups + (chunk - blk * wq.chunks_per_block) * wq.group_chunk;
      int ng = min(min(G, (blk + 1) * wq.block_groups), ga + wq.group_chunk) - ga;
      const int w0 = ng * warp / kGWarps;
      ng = ng * (warp + 1) / kGWarps - w0;
      ga += w0;
      nst = ng * stages_per_group;
      if (lane == 0) {
        it.k0 = tiles[t].k0;
        it.l0 = tiles[t].l0;
        it.row = ga * stages_per_group * kGRows;
        it.acc_off = blk * wq.block_stride + (long long)it.k0 * M + it.l0;
      }
    }
    auto issue = [&](int i) {  // lane 0: stage of step i
      const int s = (int)((qb + i) % kGSt);
      unsigned char* st = ring + (size_t)s * kGStage;
      mbar_arrive_expect_tx(&full[warp][s], kGStage);
      tma_load_2d(st, &tm32, it.k0, it.row + i * kGRows, &full[warp][s]);
      tma_load_2d(st + kGA, &tm64, it.l0, it.row + i * kGRows, &full[warp][s]);
    };
    f32x2 d[32];  // points 8 i + 2 j, 8 i + 2 j + 1 at d[4 i + j]
#pragma unroll
    for (int i = 0; i < 32; ++i) d[i] = 0ull;
    if (lane == 0)
      for (int i = 0; i < kGSt && i < nst; ++i) issue(i);
    {
      uint32_t z[16];
#pragma unroll
      for (int i = 0; i < 16; ++i) z[i] = 0u;
#pragma unroll
      for (int h = 0; h < 8; ++h) tmem_st16_g(tsum + 16 * h, z);
      tmem_wait_st_g();
    }
    __syncwarp();
    bool ok = true;
    int sg = 0;  // stage within the group
    for (int i = 0; i < nst; ++i) {
      const int s = (int)((qb + i) % kGSt);
      ok = __all_sync(0xffffffffu,
                      mbar_wait_bounded(&full[warp][s], ((qb + i) / kGSt) & 1u, status));
      if (!ok) {
        // the copies issued and not consumed land before the warp stops
        if (lane == 0)
          for (int q = i; q < nst && q < i + kGSt; ++q)
            mbar_wait_bounded(&full[warp][(qb + q) % kGSt], ((qb + q) / kGSt) & 1u, status);
        break;
      }
      const uint32_t pa = ring_s + (uint32_t)s * kGStage + 16 * tx;
      const uint32_t pb = ring_s + (uint32_t)s * kGStage + kGA + 16 * ty;
      // the rows with negative weight come first; the sum is negated where they end
      const int neg = n_neg - sg * kGRows;
      if (neg < 0 || neg >= kGRows) {
#pragma unroll
        for (int r = 0; r < kGRows; ++r) entry_row(pa + r * 128, pb + r * 256, d);
      } else {
#pragma unroll
        for (int r = 0; r < kGRows; ++r) {
          if (r == neg) {
#pragma unroll
            for (int q = 0; q < 32; ++q) {
              const float2 v = unpack2(d[q]);
              d[q] = pack2(-v.x, -v.y);
            }
          }
          entry_row(pa + r * 128, pb + r * 256, d);
        }
      }
      if (++sg == stages_per_group) {  // end of a group: c4 into the per-item sums
        sg = 0;
#pragma unroll
        for (int h = 0; h < 4; ++h) {
          uint32_t t[16];
          tmem_ld16_g(tsum + 16 * h, t);
#pragma unroll
          for (int q = 0; q < 8; ++q) {
            const float2 v = unpack2(d[8 * h + q]);
            t[2 * q] = __float_as_uint(__uint_as_float(t[2 * q]) + v.x);
            t[2 * q + 1] = __float_as_uint(__uint_as_float(t[2 * q + 1]) + v.y);
          }
          tmem_st16_g(tsum + 16 * h, t);
          tmem_ld16_g(tsum + 64 + 16 * h, t);
#pragma unroll
          for (int q = 0; q < 8; ++q) {
            const float2 v = unpack2(d[8 * h + q]);
            t[2 * q] = __float_as_uint(fmaf(v.x, v.x, __uint_as_float(t[2 * q])));
            t[2 * q + 1] = __float_as_uint(fmaf(v.y, v.y, __uint_as_float(t[2 * q + 1])));
            d[8 * h + q] = 0ull;
          }
          tmem_st16_g(tsum + 64 + 16 * h, t);
        }
        tmem_wait_st_g();
      }
      // the warp is done with stage s: its lane 0 loads the stage's next step
      __syncwarp();
      if (lane == 0 && i + kGSt < nst) {
        fence_async_smem();
        issue(i + kGSt);
      }
    }
    if (__syncthreads_or(!ok)) break;
    qb += nst;
    // end of the item: the four warps' sums of each part meet in the rings (no copy is
    // in flight), row k of the tile as 16 chunks of four columns, chunk c of row k at
    // c ^ 2 (k / 4 % 4), and a warp adds 8 rows of 64 columns to the accumulators
    float* ex = reinterpret_cast<float*>(ring);
    const int k0 = it.k0, l0 = it.l0;
    double* arow = acc + it.acc_off;
#pragma unroll 1
    for (int part = 0; part < 2; ++part) {
#pragma unroll
      for (int h = 0; h < 4; ++h) {  // points 16 h .. + 15: rows i = 2 h, 2 h + 1
        uint32_t t[16];
        tmem_ld16_g(tsum + 64 * part + 16 * h, t);
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          const int i = 2 * h + (q >> 1), r = (i >> 2) * 16 + 4 * tx + (i & 3);
          const int c = (ty + 8 * (q & 1)) ^ (2 * tx);
          *reinterpret_cast<uint4*>(ex + r * 64 + 4 * c) =
              make_uint4(t[4 * q], t[4 * q + 1], t[4 * q + 2], t[4 * q + 3]);
        }
      }
      __syncthreads();
      double* dst = arow + 2 * part * plane;  // sums, then sums of squares (real cut)
#pragma unroll 2
      for (int i = 0; i < 8; ++i) {
        const int r = 8 * warp + i, perm = 2 * ((r >> 2) & 3);
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const int l = 32 * h + lane;
          const float* col = reinterpret_cast<const float*>(ring0) + r * 64 +
                             4 * ((l >> 2) ^ perm) + (l & 3);
          if (k0 + r <= l0 + l && l0 + l < lim)
            atomicAdd(dst + (long long)r * M + l,
                      widen_sum4(col[0], col[kGRing / 4], col[2 * (kGRing / 4)],
                                 col[3 * (kGRing / 4)], wq.group_chunk <= 4));
        }
      }
      __syncthreads();
    }
    // the exchange's accesses come before the next item's copies into the ring
    fence_async_smem();
    __syncwarp();
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (warp == 0) {
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_slot),
                 "r"(kGTmemCols));
  }
}

}  // namespace

cudaError_t launch_k3_trispec_gram(const CUtensorMap& tm32, const CUtensorMap& tm64,
                                   const OperandImage& oi, int G, int m, int M, int lim,
                                   const TileInfo* tiles, int n_tiles, double* acc,
                                   long long plane, int block_groups, long long block_stride,
                                   LaunchCache* lc, unsigned* ticket, int* status,
                                   cudaStream_t stream) {
  if (G <= 0 || n_tiles <= 0) return cudaSuccess;
  if (oi.fmt != kImageGramF32 || oi.rows % kGRows != 0) return cudaErrorInvalidValue;
  const size_t smem = (size_t)kGWarps * kGRing + 1024;
  // four CTAs per SM: 128 registers a thread, 49 KB of shared memory and 128 TMEM
  // columns each
  int occ = 1;
  cudaError_t e = prepare_kernel((const void*)k3_trispec_gram, kGThreads, smem, smem, 4, lc,
                                 kSlotGram, &occ);
  if (e != cudaSuccess) return e;
  const int nsm = lc->nsm;
  WarpQueue wq;
  wq.ticket = ticket;
  wq.base = lc->drawn;
  wq.n_tiles = n_tiles;
  wq.n_combos = 1;
  if (block_groups <= 0 || block_groups > G) block_groups = G;
  wq.block_groups = block_groups;
  wq.block_stride = block_stride;
  const long long n_blocks = (G + block_groups - 1) / block_groups;
  // a group: about 100 clocks an entry row with the SM's 16 warps at work, 500 its end
  wq.group_chunk = warp_item_groups(block_groups, n_blocks * n_tiles, nsm,
                                    100.0 * oi.rows + 500.0, 2 * 2048);
  wq.chunks_per_block = (block_groups + wq.group_chunk - 1) / wq.group_chunk;
  const long long n_items = n_blocks * wq.chunks_per_block * n_tiles;
  const long long slots = (long long)occ * nsm;
  if (n_items > 0x7ffffff0ll - slots) return cudaErrorInvalidValue;
  wq.n_items = (int)n_items;
  const int n_cta = (int)std::min(slots, n_items);
  lc->drawn += (unsigned)(n_items + n_cta);
  k3_trispec_gram<<<n_cta, kGThreads, smem, stream>>>(tm32, tm64, oi.rows / kGRows,
                                                      m * (m - 1) / 2 + 1, G, M, lim, tiles, wq,
                                                      acc, plane, status);
  return cudaGetLastError();
}

}  // namespace ss
