// internal.cuh -- definitions shared by the kernels and the host runtime of the
// polyspectrum library (not part of the public ABI; see include/polyspec.h).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include <string>
#include <vector>

#include "pipeline.cuh"
#include "polyspec.h"

namespace ss {

// Size of the static scratch array of ss_s2_noalloc.
constexpr size_t kNoallocScratchBytes = SS_NOALLOC_SCRATCH_BYTES;

// Tile edge of the bispectrum and trispectrum kernels in (k, l) grid points.
// shared memory of the resident form of K1 (group coefficients + FFT batch)
constexpr size_t kK1ResidentBytes = 96u << 10;
// a tighter budget tried first: three resident CTAs per SM
constexpr size_t kK1ResidentBytes3 = 74u << 10;
constexpr int kTile = 64;
// Largest frame length and channel count a plan takes (the kernels' fixed
// dynamic shared-memory limits are sized for them).
constexpr int kMaxT = 4096, kMaxChannels = 4;
// Largest frames per staged chunk of the pair kernels.
constexpr int kMaxFC = 16;
// Threads per CTA of the frame/FFT kernel and of the pair kernels.
constexpr int kThreadsK1 = 256;
constexpr int kThreadsPair = 256;

// Accumulator planes per grid point: sum Re S_g, sum Im S_g, sum (Re S_g)^2,
// sum (Im S_g)^2, all float64 (Sec. 4.2, Eq. 35-36 need the first and second
// power sums over the parts).
constexpr int kPlanes = 4;

// Where the samples of one batch come from: the plan's carry-over buffer
// (samples left from earlier chunks) followed by the caller's chunk.  Sample s
// of channel c in the concatenated record is carry[c*carry_stride + s] for
// s < carry_n and chunk[c*chunk_stride + s - carry_n] otherwise.
struct SampleSource {
  const void* carry;
  long long carry_n;
  long long carry_stride;
  const void* chunk;
  long long chunk_stride;
  int dtype;  // SS_F32 or SS_I16
};

// Groups of a block when a batch is one block (its sums in one place).
constexpr int kOneBlock = 0x7fffffff;

// The centred spectra K1 writes: bin 0 of channel c's frame row r is at
// rows + c * chan_stride + r * stride.  Mp bins from there on are written (zeros
// past M - 1); with mirror, also the conjugates at the bins -(M - 1) .. -1 before.
// Without store, nothing reads the spectra (S2 alone) and they need not be written.
// The S2 sums of block g / block_groups of the groups go block_stride doubles apart.
struct SpecRows {
  float2* rows;
  long long chan_stride;
  int stride, mirror, store;
  int block_groups = kOneBlock;
  long long block_stride = 0;
};

// One channel combination of one order; channels as in the ABI records.
struct Combo {
  int order;
  int c[4];
};

// Optional second output of K1 for the tensor-core S4 kernel: the operand
// image of the weighted frame Gram of every bin.  With centred coefficients d_j
// of a group, G_jj' = Re(d_j d_j'*), the bracket of the factorised fourth
// k-statistic (App. H, Eq. 85) for the cut (a_k, a_k*, a_l, a_l*) is
//   m(m+1) Q - (m-1)(|U|^2 + |V|^2) = sum_{j<=j'} w_jj' G^k_jj' G^l_jj',
//   w_jj = m^2 - m + 2,  w_jj' = -4(m-1) (j < j'),
// one real contraction over K = m(m+1)/2, and c4 = r [that - (m-1) Sk Sl] with
// r = 1/((m-1)(m-2)(m-3)), Sk = sum_j |d_jk|^2.  The K entries come in chunks
// of 16: the diagonal chunks first, scaled by sd = sqrt(w_jj r), then the pairs
// j < j' in lexicographic order, scaled by so = sqrt(4(m-1) r), then one entry
// ps_k = sp Sk, sp = sqrt((m-1) r), zero-padded (the tensor-core kernel negates
// the pair chunks, so ps_k ps_l is subtracted with them and the contraction is
// c4 itself; K = m(m+1)/2 + 1).  Each entry is split hi + lo.  Layout per
// channel and group: rows (bins) in groups of 8; per row group, for each chunk,
// a hi block and a lo block of CB bytes, each holding the row group's core
// matrices (8 rows x 16 bytes) of the chunk's 16-byte entry groups 128 bytes
// apart (TF32: CB = 512; BF16, FP16: CB = 256).  So a chunk of a row group is
// 2 CB bytes, a row group rg_bytes = nkc * 2 CB, a group group_bytes =
// (Mp / 8) * rg_bytes.
// FP16: each bin's row is first multiplied by a power of two s_k that brings its
// largest entry (at most max(max(sd, so) max_j |d_jk|^2, sp Sk)) below 2^14, so
// that hi and lo stay inside the FP16 range; rsc holds 1/s_k per group and bin,
// and the kernel divides D by s_k and by s_l (exactly: powers of two).
// F32 (k3_trispec_gram, CUDA cores): the entries unsplit and unscaled, one row of Mp
// bins per entry, rows rows a group: the pairs, ps, the diagonal, then zeros up to a
// multiple of kGram32Rows.
enum { kImageNone = 0, kImageGramTF32 = 1, kImageGramBF16 = 2, kImageGramF16 = 3,
       kImageGramF32 = 4 };
constexpr int kGram32Rows = 8;   // entry rows of a stage of k3_trispec_gram
// Largest m of k3_trispec_gram; K1 and S4 with it against k3_trispec at T = 1024, 2^24
// samples (ms): m = 5 0.58 / 1.56, 10 0.72 / 1.21, 14 0.91 / 1.13, 16 0.99 / 1.09 (m = 17
// with k3_trispec 1.24).
constexpr int kGram32MaxM = 16;
constexpr int kMaxGramM = 32;  // largest m of the tensor-core S4 path
struct OperandImage {
  void* img = nullptr;
  float* rsc = nullptr;       // FP16: per group and bin, 1 / the bin's row scale
  int fmt = kImageNone;
  int nkc = 0, ndc = 0;       // K chunks, of which diagonal
  int rows = 0;               // F32: entry rows of a group
  float sd = 0.f, so = 0.f, sp = 0.f;
  long long rg_bytes = 0;     // nkc * 2 * CB
  long long group_bytes = 0;  // (Mp / 8) * rg_bytes
  long long chan_bytes = 0;   // Gb_max * group_bytes
  long long chan_rsc = 0;     // Gb_max * Mp floats (FP16)
  int img_bins = 0;           // bins whose image rows and scales the tensor-core S4 reads
                              // (M - 1 when k3_column takes the last column, else Mp)
  // several channels in FP16X3: per channel, group and bin the power of two that
  // brings the bin's coefficients over the group's frames below 2^14 (within
  // [2^-60, 2^60]; 1 for a zero bin), at rmax[channel * chan_rmax + group * Mp + bin]
  float* rmax = nullptr;
  long long chan_rmax = 0;
};

// K1 forms (the autotuner's choice per plan): groups resident in shared memory
// within 74 KB (three CTAs per SM) when they fit, else 96 KB (kK1Auto); always
// the 96 KB budget (kK1Resident96); one frame at a time (kK1Frames); resident
// groups with a warp per frame (kK1Warp, T <= 1024 and the group within 96 KB).
enum { kK1Auto = 0, kK1Resident96 = 1, kK1Frames = 2, kK1Warp = 3, kK1Modes = 4 };

// What a plan keeps between launches: the GPU's SM count, for each kernel whether its
// function attributes are set and how many CTAs an SM holds of it with this plan's
// shared memory (0: not asked yet), and how many items the plan's kernels have drawn
// from its ticket counter since the last reset (the counter runs on, so a launch needs
// no memset: its items are the tickets from there on).  A launch without one asks the
// runtime each time.
enum { kSlotK1Res74 = 0, kSlotK1Res96, kSlotK1Warp, kSlotK1Frames, kSlotK1Power, kSlotK1Fft,
       kSlotK1Centre, kSlotK2Warp, kSlotGram, kSlotTc, kSlots };
struct LaunchCache {
  int nsm = 0;
  int occ[kSlots] = {};
  unsigned drawn = 0;
};
// Set a kernel's shared-memory attributes (one fixed limit per kernel, whatever launch
// comes first) and find its resident CTAs per SM from its registers and shared memory
// (the occupancy query reports fewer for some of these kernels than both limits allow),
// at most max_ctas; both once per cache.
cudaError_t prepare_kernel(const void* kern, int threads, size_t smem, size_t limit, int max_ctas,
                           LaunchCache* lc, int slot, int* occ);
cudaError_t sm_count(LaunchCache* lc, int* nsm);

// Radix of the next pass of K1's Stockham transform with `rem` still to go (N = T/2 is
// a power of two).
__host__ __device__ inline int fft_radix(int rem) {
  return rem % 8 == 0 && rem != 16 ? 8 : rem % 4 == 0 ? 4 : 2;
}
// K1's twiddles, e^{+2 pi j a/T} at a = twiddle_angle(T, i) for entry i: first a = 0 ..
// N/2 (the split into the real frame's coefficients), then per pass of radix R over
// sub-transforms of length Ns > 1 the factors r k T/(Ns R), r = 1 .. R - 1, as R - 1
// rows of Ns entries k, so that a warp's loads are consecutive.  (Indexed by r k T/(Ns R)
// in one table of T entries, a warp's 7 loads of a radix-8 pass fell on one bank up to
// 16 times: most of the passes' shared-memory time.)
inline __host__ __device__ int twiddle_count(int T) { return (3 * T / 4 + 2) & ~1; }
inline __host__ __device__ int twiddle_angle(int T, int i) {
  const int N = T / 2;
  if (i <= N / 2) return i;
  int off = N / 2 + 1, Ns = 1;
  for (int rem = N; rem > 1;) {
    const int R = fft_radix(rem);
    if (Ns > 1) {
      const int cnt = (R - 1) * Ns;
      if (i < off + cnt) return ((i - off) / Ns + 1) * ((i - off) % Ns) * (T / (Ns * R));
      off += cnt;
    }
    Ns *= R;
    rem /= R;
  }
  return 0;  // padding
}

// Kernel launchers (each returns the launch status; all work on `stream`).
cudaError_t launch_k1_spectra(const SampleSource& src, long long sample0, int G, int C, int T,
                              int m, int M, int Mp, const float* win, const float2* tw,
                              const SpecRows& spec, const int* s2_auto, double* acc2, int n_s2,
                              float pref2, LaunchCache* lc, cudaStream_t stream,
                              const OperandImage& oi = OperandImage(), double* acc1 = nullptr,
                              int mode = kK1Auto);

cudaError_t launch_k1_cross_s2(const float2* spec, long long chan_stride, int G, int m, int M,
                               int Mp, const int4* pairs, int n_pairs, float pref2, double* acc2,
                               long long plane, int nsm, cudaStream_t stream);

// Pair kernels run persistent grids of nsm x (resident CTAs per SM) CTAs that
// take (group chunk, tile) items from a queue (see pipeline.cuh); `counter` is
// a device int the launcher zeroes on the stream.  acc points at the
// combination's first accumulator plane; `plane` is the distance in doubles
// between the four planes (sum Re, sum Im, sumsq Re, sumsq Im).  `status` is
// the plan's device status word (a bounded wait that gives up writes to it);
// inject_timeout != 0 makes K2 run one wait out on purpose (timeout test).
// The tensor maps view the centred spectra as [rows][Mp/16][16] float2 with
// 128-byte swizzling; tm64 has boxes of 4 blocks (64 bins), tm128 of 8.
// K2 tilings (the autotuner's choice per plan): 4 x 4 micro-tiles in CTAs of 256
// threads with 4 stages (two CTAs per SM) or 3 stages (three CTAs per SM, 85
// registers), or 8 x 4 micro-tiles in CTAs of 128 threads with 2 or 3 stages;
// all take the same 64 x 64 tiles and give the same sums.  kK2Warp84, the default, runs
// k2_bispec84w: 8 x 4 micro-tiles on 32 x 32 sub-tiles, a ring of stages per warp.
enum { kK2Tile44 = 0, kK2Tile84Stages2 = 1, kK2Tile84Stages3 = 2, kK2Tile44Stages3 = 3,
       kK2Warp84 = 4, kK2Variants = 5 };
cudaError_t launch_k2_bispec(const CUtensorMap& tm64, const CUtensorMap& tm128,
                             const float2* spec_a, const float2* spec_b, const float2* spec_c,
                             int rowA, int rowB, int rowC, int G, int m, int FC, int M, int Mp,
                             const TileInfo* tiles, int n_tiles, int cross, float pref3,
                             double* acc, long long plane, int rows, int nsm, int* counter,
                             int* status, int inject_timeout, int variant, cudaStream_t stream);

cudaError_t launch_k3_trispec(const CUtensorMap& tm64, int row0, int G, int m, int FC, int M,
                              const TileInfo* tiles, int n_tiles, float pref4a, float pref4b,
                              double* acc, long long plane, int nsm, int* counter, int* status,
                              cudaStream_t stream);

// The FP32 form for groups of at most kGram32MaxM frames: K1's F32 operand image
// through 2-D views [group x rows][Mp] with boxes of 32 (tm32) and 64 (tm64) bins x
// kGram32Rows rows; tiles of 32 x 64 (k, l) bins below lim, sums stored at [k][l].
// Blocks of groups as for launch_k2_bispec84w.
cudaError_t launch_k3_trispec_gram(const CUtensorMap& tm32, const CUtensorMap& tm64,
                                   const OperandImage& oi, int G, int m, int M, int lim,
                                   const TileInfo* tiles, int n_tiles, double* acc,
                                   long long plane, int block_groups, long long block_stride,
                                   LaunchCache* lc, unsigned* ticket, int* status,
                                   cudaStream_t stream);

// Tensor-core form of K3 (SS_PREC_TF32X3, SS_PREC_BF16X3, SS_PREC_BF16): tiles of
// 128 x 128 (k, l) bins, the weighted frame-Gram contraction fed from K1's
// operand image of `channel` through tm_img, a 4-D view of that channel's
// image [group][row group][chunk][2 CB bytes] in 8-byte elements with boxes of
// k3tc_stage_chunks(precision) chunks x 16 row groups; needs 4 <= m <= kMaxGramM.
constexpr int kTcTileM = 128, kTcTileN = 128;
cudaError_t launch_k3_trispec_tc(const CUtensorMap& tm_img, const OperandImage& oi, int channel,
                                 int G, int m, int M, int Mp,
                                 const TileInfo* tiles, int n_tiles, int precision, double* acc,
                                 long long plane, int block_groups, long long block_stride,
                                 LaunchCache* lc, unsigned* ticket, int* status,
                                 cudaStream_t stream);
size_t k3tc_smem_bytes(int precision);

// K3 for several channels (FP32 CUDA cores): C4(a_k, b_k*, c_l, d_l*) of every
// combination (combos: device array of n_combos (a, b, c, d)) on the grid
// k in [-(M-1), M-1] x l in [0, M-1], accumulated at acc[plane][combo][k+M-1][l].
// A combination with a == b or c == d is symmetric: exchanging x and y (a == b) or z
// and w together with the conjugation of all four (c == d) gives
//   S4(-k, l) = S4(k, l) (a == b),  S4(-k, l) = S4(k, l)* (c == d),
// so only its rows k >= 0 are computed and mirrored (34 of 55 combinations of four
// channels).  rowtiles: device array of n_rowtiles (combination, first row r = k + M - 1);
// half: device array of n_half (combination, 1 to conjugate) of the mirrored ones.
constexpr int kCrossRows32 = 32;  // rows and columns of a tile of the FP32 kernel
struct CrossTiles {
  const int2* rowtiles = nullptr;
  const int2* half = nullptr;
  int n_rowtiles = 0, n_half = 0;
};
cudaError_t launch_k3_trispec_cross(const float2* spec, long long chan_stride, int G, int m, int M,
                                    int Mp, const int4* combos, int n_combos, const CrossTiles& ct,
                                    double* acc, long long plane, int nsm, bool natural,
                                    cudaStream_t stream);
// the row k = M - 1 of the mirrored combinations, in FP32
cudaError_t launch_k3_cross_last_row(const float2* spec, long long chan_stride, int G, int m, int M,
                                     int Mp, const int4* combos, const CrossTiles& ct, float pref,
                                     float fmm, float fm1, double* acc, long long plane,
                                     cudaStream_t stream);
// rows k < 0 of the mirrored combinations from the rows k > 0 (by assignment, after
// every batch), and with row0 also the row k = -(M - 1) of the others from k = M - 1
cudaError_t launch_k3_cross_mirror(const CrossTiles& ct, int n_combos, int M, double* acc,
                                   long long plane, bool row0, cudaStream_t stream);
int k3tc_stage_chunks(int precision);

// The same on the tcgen05 tensor cores: tiles of 128 rows k x 24 columns l,
// operands built in shared memory from the centred spectra.  TF32 hi/lo in three
// passes for SS_PREC_TF32X3, SS_PREC_BF16X3 and SS_PREC_BF16; with SS_PREC_FP16X3
// FP16 hi/lo in three passes of operands scaled per bin by powers of two, the
// bins' row scales per group that K1 writes (OperandImage::rmax).
// The spectra are read through 2-D views [rows][Mp] (8-byte elements, no swizzle):
// tm_ab with boxes of kF rows x min(box bins, Mp) bins, tm_cd with boxes of kF
// rows x col box bins (kF = 4 frames, 8 for FP16); a channel's rows start at
// channel x chan_rows; spec, chan_stride and Ms address the same coefficients.  The
// mirrored combinations' row k = M - 1, alone in its tile where M - 1 is a multiple of
// 128, is left to a CUDA-core kernel.  FP16 also reads the row scales [channel x grp_rows +
// group][Mp] (float) through tm_sab (boxes of min(kCrossScaleBins, Mp) bins) and
// tm_scd (kCrossScaleCols bins).  The row k = -(M-1) is copied from k = M-1 (equal
// for real signals).  counter and status as for the pair kernels.
// Box widths (bins) of tm_ab and tm_cd, TF32 and FP16 forms: wider than the bins
// used, so that the rows of a thread's two frame chunks fall on other banks.
constexpr int kCrossBoxBins = 140, kCrossBoxBinsH = 142, kCrossColBox = 28, kCrossColBoxH = 30;
constexpr int kCrossTileRows = 128, kCrossTileCols = 24, kCrossScaleBins = 144, kCrossScaleCols = 28;
struct CrossViews {
  const CUtensorMap* tm_ab = nullptr;
  const CUtensorMap* tm_cd = nullptr;
  const CUtensorMap* tm_sab = nullptr;
  const CUtensorMap* tm_scd = nullptr;
  int chan_rows = 0, grp_rows = 0;
  bool f16 = false;
};
cudaError_t launch_k3_trispec_cross_tc(const CrossViews& v, int G, int m, int M, int Mp,
                                       const int4* combos, int n_combos, const CrossTiles& ct,
                                       const float2* spec, long long chan_stride, int Ms,
                                       double* acc, long long plane, int nsm, bool natural,
                                       int* counter, int* status, cudaStream_t stream);

// Most groups whose per-group estimates a kernel adds up in float32 before the
// run goes to the float64 accumulators (bounds the float32 rounding of the sums
// over groups of Sec. 4.2 whatever the record length).
constexpr int kMaxFp32Groups = 64;

// Groups per work item: about 16 items per CTA, whole groups, at least one, at
// most kMaxFp32Groups (the pair kernels sum an item's groups in float32).
inline int work_group_chunk(int G, int n_tiles, int n_cta) {
  const long long units = (long long)G * n_tiles;
  const long long target = 16ll * n_cta;
  long long gc = (units + target - 1) / target;
  if (gc < 1) gc = 1;
  if (gc > kMaxFp32Groups) gc = kMaxFp32Groups;
  if (gc > G) gc = G;
  return (int)gc;
}

// Runs of groups of k3_trispec_cross and K5, of at most kMaxFp32Groups groups: CTAs for
// one full wave of kRunCtas per SM where that leaves at most a seventh of the places
// empty, else for four waves.
constexpr int kRunCtas = 3;
inline int group_runs(int G, long long ctas_per_run, int nsm) {
  const long long places = (long long)kRunCtas * nsm;
  long long runs = places / ctas_per_run;
  if (runs * ctas_per_run * 7 < places * 6) runs = (4 * places + ctas_per_run - 1) / ctas_per_run;
  runs = std::max(runs, (long long)(G + kMaxFp32Groups - 1) / kMaxFp32Groups);
  runs = std::min<long long>(std::min<long long>(runs, G), 65535);
  return (int)std::max(1ll, runs);
}

// Spectra of complex-valued signals (App. D) and shifted S4 planes (App. E) on
// the full (k, l) plane: n_combos combinations of `order` operands each, operand
// i of combination q at ops[order q + i] = (real channel, imaginary channel or
// -1, sign of j: -1 for the conjugate signal, else 1); accumulated at
// acc[plane][q][rows][cols] with rows = cols = 2M - 1 (S2: [q][2M - 1]).
cudaError_t launch_k5_complex(const float2* spec, long long chan_stride, int G, int m, int M,
                              int Mp, int order, const int4* ops, int n_combos, int shift,
                              bool natural, double* acc, long long plane, int nsm,
                              cudaStream_t stream);

// Groups of an item of k2_bispec84w or k3_trispec_gram, for blocks of G groups times
// `tiles` (tiles, combinations and blocks).  Estimated, in clocks: a group takes a warp
// `group` with the SM full, up to 1.75 times that with fewer items on an SM than it
// holds; an item 1500 more; the last items of an SM end unevenly; and the `adds`
// float64 additions of an item are taken by the L2 at about 200 a clock over the whole
// GPU.  A warp takes a quarter of the groups, at most kMaxFp32Groups.  Measured (ms, K2 alone) for
// 4 / 8 / 16 / 64 groups: T = 1024, m = 10, 2^28 samples 10.21 / 8.20 / 7.34 / 6.75;
// T = 128, m = 32, 2^23 samples 0.113 / 0.108 / 0.130 / 0.166; T = 256, m = 10, 2^20
// samples 0.033 / 0.033 / 0.040 / 0.062.
inline int warp_item_groups(int G, long long tiles, int nsm, double group, int adds) {
  int best = 1;
  double tb = 1e300;
  const int top = G < 4 * kMaxFp32Groups ? G : 4 * kMaxFp32Groups;
  for (int gc = 1; gc <= top; ++gc) {
    const long long items = (long long)((G + gc - 1) / gc) * tiles;
    const double item = ((gc + 3) / 4) * group + 1500.0;
    const long long full = (items + nsm - 1) / nsm;  // items of the busiest SM
    const double rounds = full == 1   ? 1.75
                          : full == 2 ? 2 * 1.5
                          : full == 3 ? 3 * 1.3
                          : full == 4 ? 4 * 1.1
                                      : (double)items / nsm + 1.0;
    const double t = rounds * item + (double)items * (adds / 200.0);
    if (t < tb) {
      tb = t;
      best = gc;
    }
  }
  return best;
}

// Independent warps on 32 x 32 sub-tiles, every combination in one launch: combos
// is a device array of n_combos channel triples (x, y, z) whose sums start
// combo_stride doubles apart; channel c's rows start at c * chan_rows.  tm32 /
// tm64w: boxes of 2 / 4 blocks (32 / 64 bins) x kFrames84w frame rows of the
// spectra, bin 0 in block zblk of a row.  One channel: the plan's list of
// sub-tiles with more than 8 points of the domain (k2_points takes the others'
// points) or of all; several: every sub-tile that touches the domain.  Groups form
// blocks of block_groups (0: one block) whose sums are block_stride doubles apart.
constexpr int kFrames84w = 4;
cudaError_t launch_k2_bispec84w(const CUtensorMap& tm32, const CUtensorMap& tm64w, int chan_rows,
                                int zblk, int G, int m, int M, const TileInfo* tiles, int n_tiles,
                                const int4* combos, int n_combos, int cross, float pref3,
                                double* acc, long long plane, long long combo_stride,
                                int block_groups, long long block_stride, LaunchCache* lc,
                                unsigned* ticket, int* status, int inject_timeout,
                                cudaStream_t stream);
// K2 for isolated grid points of one channel (pts: n_pts (k, l) pairs)
cudaError_t launch_k2_points(const float2* spec, int Mp, int G, int m, const int2* pts,
                             int n_pts, int M, float pref3, double* acc, long long plane,
                             cudaStream_t stream);

// the one-channel S4 cut at l = M - 1 for every k, stored at acc[k * sk + l * sl]
cudaError_t launch_k3_column(const float2* spec, int Mp, int G, int m, int M, float pref4a,
                             float pref4b, double* acc, long long plane, int sk, int sl,
                             int block_groups, long long block_stride, cudaStream_t stream);

// dynamic shared memory of the pair kernels for FC frames per stage
size_t k2_smem_bytes(int FC);
size_t k3_smem_bytes(int FC);

// K4: mean and standard error over G groups of the float64 sums in acc, or, with
// prev, of the sums acc - prev (the groups since a snapshot: sequential spectra).
cudaError_t launch_k4_finalize(const double* acc, int n_combos, int rows, int M, int layout,
                               long long G, double norm, double* out, double* err,
                               cudaStream_t stream, const double* prev = nullptr);

// Several grids in one launch, and n_blocks sets of them: set y reads the sums
// acc_stride y doubles on and writes out_stride y doubles on.  Either of out and err
// (device memory) may be NULL; launch_k4 drops grids with neither.
struct K4Job {
  const double* acc;
  const double* prev;
  double* out;
  double* err;
  long long plane, acc_stride, out_stride;
  double mean_scale, sq_scale, mean_sq_scale;
  int n_combos, rows, M, layout, first_block, wide;
};
constexpr int kK4Jobs = 3;
struct K4Jobs {
  K4Job job[kK4Jobs];
  int n;
};
K4Job k4_job(const double* acc, int n_combos, int rows, int M, int layout, long long G, double norm,
             double* out, double* err, const double* prev = nullptr);
cudaError_t launch_k4(K4Jobs& js, int n_blocks, cudaStream_t stream);

// acc[i] += the sum over n_blocks of blk[b * stride + i], and prev[i] = acc[i], i < n
cudaError_t launch_add_blocks(double* acc, double* prev, const double* blk, long long stride,
                              int n_blocks, long long n, cudaStream_t stream);

// dst[i] += src[i], i < n (device pointers): merges exported group sums.
cudaError_t launch_add_f64(double* dst, const double* src, long long n, cudaStream_t stream);

// Layout codes of launch_k4_finalize.
enum { kLayoutVector = 0,       // S2: [M]
       kLayoutS3Single = 1,     // one channel, computed for k <= l, mirrored; k+l <= M-1
       kLayoutS4Single = 2,     // one channel, computed for k <= l, mirrored
       kLayoutCross = 3,        // full [2M-1][M] grid, no mirroring
       kLayoutS4Lower = 4 };    // one channel, point (k, l), k <= l, stored at [l][k]

}  // namespace ss
