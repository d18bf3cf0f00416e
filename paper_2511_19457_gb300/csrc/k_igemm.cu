// Dense and zero-skipping implicit-GEMM kernel on the 5th-generation tensor
// cores (tcgen05, accumulators in tensor memory), sm_103a.
//
// Persistent: one CTA per SM walks the output tiles (128 rows x BN columns)
// of y = epilogue(A * B^T) with a static round-robin schedule.  Two tensor-
// memory accumulators (lean kernels up to 128 columns wide: four) alternate
// between tiles, so the epilogue of tile i (TMEM -> registers -> swizzled shared
// memory -> TMA store) overlaps the MMAs of tile i + 1, and the shared-memory
// stage ring never drains between tiles.
//
// B [N, K] holds the weights (K-major; [C_out][kh][kw][C] for a convolution)
// and is loaded by TMA.  A (128 rows of K) comes in one of three ways:
//   mode 0  GEMM: A = x[M, K] row-major; rows m0..m0+127; 2-D TMA box.
//   mode 2  convolution, C % BK == 0: the 128 rows are a spatial output tile
//           of bw x bh pixels in bn images; for K block (tap r,s; BK channels)
//           one 4-D TMA box {BK channels, bw, bh, bn} of the NHWC input at the
//           shifted, strided origin (element strides = conv stride) is the A
//           tile; out-of-range coordinates read zeros, which is the padding.
//   mode 1  convolution, any C % 8 == 0: 128 consecutive output pixels,
//           gathered by 128 producer threads with cp.async.
//   stem    C < 8 (the RGB input), N <= 64: 128 consecutive output pixels, built
//           in shared memory from the input rows ([32,224,224,3] 7x7/2 -> 64 with
//           statistics and occupancy: 103 -> 60 us a call; im2col rows in memory
//           cost 44 us to write and 26 us to read back).
// K advances in BK-wide blocks: BK = 64 with the 128-byte swizzle (four
// tcgen05.mma of K = 16 per stage) or BK = 32 with the 64-byte swizzle.
//
// Threshold dispatch (Sec. 3 rule, thresholds as parameters) is evaluated in
// the kernel prologue from the input's Eq. 1 count, so no host round trip
// separates statistics and compute.  On the zero-skip path each tile leaves
// out the K blocks whose activations are all zero over its 128 rows (Sec. 2.1:
// products with zero activations can be skipped without changing the result):
//   GEMM: from the 128-row block-column mask of x (one word per 32 columns);
//   conv: from the row bitmaps of the tile's shifted input pixels, reduced
//         per tile into a per-tap mask of occupied 64-channel tiles.
// The epilogue applies bias / batch norm / residual / activation, stores y and
// writes y's Eq. 1 count and occupancy bitmaps for the next operator.
//
// Warp roles: producer warps (the skip masks; one lane of warp 0 issues TMA; in
// mode 1 all 128 threads gather, in stems all seven warps build), epilogue warps
// from warp 4 (stems: 8) on by TMEM lane quarter, each taking 32-column blocks,
// one warp for TMEM allocation and MMA issue.
//
// Each tile shape is compiled three times: the general kernel (mode 1, fp32
// output, the dense half of a small FC), and lean ones for modes 0 and 2 with
// bf16 output, without a residual and with one (N % 8 == 0).  Small-K problems are bound by the epilogue's latency
// and by what feeds it, so the lean kernel has 16 epilogue warps that never wait
// for each other, four accumulators in flight (up to 128-wide tiles), one
// converged producer warp that lays out 32 tiles at a time, and keeps weights
// that fit the ring.  Measured (GB300, BN + ReLU6 + output occupancy): the 1x1
// expansion [32,112,112,16] -> 96 53.5 -> 34.5 us (90 MB: 2.6 TB/s; 22.9 without
// the occupancy), [32,56,56,24] -> 144 35.9 -> 22.9 us, the MLP's up projection
// [6304,768] x [3072,768] + GELU 48 -> 34 us.  One column block's instructions
// appear once: a second copy (planes of two blocks in registers) cost the wide
// tiles 10 % in instruction-cache misses.
#include <cuda.h>
#include <cudaTypedefs.h>


#include <mutex>

#include "igemm_geo.cuh"
#include "sparoa_kernels.h"

namespace sparoa {

namespace {

constexpr int kMaxSplit = 4;  // K split: at most this many units per output tile
// Warp roles.  The general kernel: 4 producer warps (all 128 threads gather in
// mode 1), 8 epilogue warps (two per TMEM lane quarter), the MMA warp.  The
// lean ones: 3 producer warps, the MMA warp, 16 epilogue warps -- 5 warps per
// scheduler, which leaves 96 registers a thread (a 21st warp would leave 80 and
// spill).  Stems, whose producers build the A tiles: 7 producer warps, the MMA
// warp, 8 epilogue warps.
template <int LEAN, bool STEM = false>
struct Warps {
  static constexpr int kProd = STEM ? 7 : LEAN ? 3 : 4;
  static constexpr int kEpi = LEAN && !STEM ? 16 : 8;
  static constexpr int kEpiThreads = 32 * kEpi;
  static constexpr int kEpi0 = STEM ? 8 : 4;  // first epilogue warp (a multiple of 4: its lane quarter)
  static constexpr int kMma = STEM ? 7 : LEAN ? 3 : kEpi0 + kEpi;
  static constexpr int kThreads = 32 * (STEM ? 16 : LEAN ? 20 : 13);
};
constexpr int kMaxKWords = 128;  // K-block occupancy bits: up to 4096 blocks
constexpr int kMaxTaps = 64;
constexpr int kStgBytes = 2 * 128 * 128;  // output staging: 32 rows x 64 bytes per epilogue warp (two each in the general kernel)
constexpr int kWarpStgBytes = 32 * 64;
constexpr int kMaxAccColsGemm = 4096;  // per-CTA column counters (output occupancy)
constexpr int kMaxStemRows = 48;      // input rows staged per tile (stem)
constexpr int kStemRowBytes = 24 * 1024;  // ... and their bytes, per buffer

// STEM: a stage is the whole A tile (three 64-wide K blocks), two of them; the
// weights' three K blocks stay; two buffers of staged input rows follow.
template <int BN, int BK, bool STEM = false>
struct Cfg {
  static constexpr int kMaxAccCols = STEM ? 64 : kMaxAccColsGemm;
  static constexpr int kAStage = (STEM ? 3 : 1) * kBM * BK * 2;
  static constexpr int kBStage = BN * BK * 2;
  static constexpr int kStageBytes = kAStage + kBStage;
  // Stage ring: about 200 KB of shared memory in all; a deeper ring made the
  // latency-bound small GEMMs and convs slower on GB300 (256 x 3072 x 768:
  // 13.6 -> 16.4 us).  192-wide tiles take all of the 227 KB for a fourth
  // 40 KB stage (4096 x 3072 x 768: 26.1 -> 22.3 us).  kFixed is everything
  // but the ring (barriers and flags of at most 12 stages) plus the 1024 bytes
  // of alignment slack.
  // column affine: general kernel scale[2][BN], shift[2][BN]; lean kernels
  // scale[BN], shift[BN] and 64 floats per epilogue warp
  static constexpr int kAffBytes = 4 * BN * 4 > 2 * BN * 4 + 16 * 256 ? 4 * BN * 4 : 2 * BN * 4 + 16 * 256;
  static constexpr int kFixed = kStgBytes + (2 * 12 + 10) * 8 + (12 + 8) * 4 + 16 + kMaxKWords * 4 +
                                kMaxTaps * 8 + kAffBytes + 4 * BN * 4 + kMaxAccCols * 4 + kBM * 8 +
                                (BN / 32) * 4 + 16 + 1024;
  static constexpr int kBudget =
      BN == 192 ? 227 * 1024 - kFixed : 200 * 1024 - kStgBytes - 6 * 1024 - kMaxAccCols * 4;
  static constexpr int kStagesRaw = kBudget / kStageBytes;
  static constexpr int kStages = STEM ? 2 : kStagesRaw > 12 ? 12 : kStagesRaw;
  static constexpr int kLag = kStages - 2;  // cp.async stages in flight (mode 1)
  static constexpr int kAOff = 0;
  static constexpr int kBOff = kAOff + kStages * kAStage;
  static constexpr int kStgOff = kBOff + (STEM ? 3 : kStages) * kBStage;  // 1024-aligned
  static constexpr int kBarOff = kStgOff + kStgBytes;
  static constexpr int kNumBars = 2 * kStages + 10;                  // full, empty, accf[4], acce[4], drain, resident B
  static constexpr int kFlagOff = kBarOff + kNumBars * 8;
  static constexpr int kKBitsOff = (kFlagOff + (kStages + 8) * 4 + 15) & ~15;
  static constexpr int kTapOff = kKBitsOff + kMaxKWords * 4;
  static constexpr int kScaleOff = kTapOff + kMaxTaps * 8;
  static constexpr int kCntOff = kScaleOff + kAffBytes;
  static constexpr int kAccOff = kCntOff + 4 * BN * 4;
  static constexpr int kRowOff = kAccOff + kMaxAccCols * 4;   // [128] row bits of the tile (general kernel)
  static constexpr int kBlkOff = kRowOff + kBM * 8;           // [BN / 32] block-mask words (general kernel)
  // [16 warps][BN / 32 blocks][3 planes][32] bit-sliced column counts (lean, BN <= 128)
  static constexpr int kPlaneOff = (kBlkOff + (BN / 32) * 4 + 15) & ~15;
  static constexpr int kPlaneBytes = BN <= 128 ? 16 * (BN / 32) * 3 * 128 : 0;
  // staged input rows [2][kStemRowBytes], per-tile tables [2]: row origins, pixel offsets
  static constexpr int kStemOff = (kPlaneOff + kPlaneBytes + 127) & ~127;
  static constexpr int kStemTabOff = kStemOff + 2 * kStemRowBytes;
  static constexpr int kStemTab = kMaxStemRows * 4 + kBM * 4;
  static constexpr int kBytes = STEM ? kStemTabOff + 2 * kStemTab : kPlaneOff + kPlaneBytes + 16;
  static constexpr int kSmem = kBytes + 1024;  // slack for 1024-byte alignment
  // TMEM: accumulator b starts at column b * kAccCols (BN rounded up to a
  // power of two, so each starts on a power-of-two column; stems: two halves);
  // the allocation covers all of them
  static constexpr uint32_t kAccCols = BN <= 64 ? (STEM ? 128u : 64u) : (BN <= 128 ? 128u : 256u);
  static_assert(kStages >= 2, "stages");
  static_assert(kSmem <= 227 * 1024, "shared memory");
};

// One row's 32 accumulator values (fp32 bits) through the column affine
// (scale and shift from shared memory; none when sc is null), the residual
// (bf16 at rp, none when rp is null; only the first rvalid of the 32 columns
// are read, rvalid a multiple of 8) and the activation, packed to 16 bf16
// pairs: fp32x2 FMAs, ReLU folded into the conversion.  The same operations
// in the same order as the general epilogue (fmaf, then + residual, then the
// activation, then round to bf16).
template <int ACT, bool RES>
__device__ __forceinline__ void affine_act_pack32(const uint32_t (&raw)[32], const float* sc, const float* sh,
                                                  const uint4* rp, int rvalid, uint32_t (&pk)[16]) {
  uint4 rv = make_uint4(0u, 0u, 0u, 0u);  // residual values 8 (i / 2) .. + 7
  if (!RES) rp = nullptr;
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    if (RES && rp && (i & 1) == 0) rv = 8 * (i >> 1) < rvalid ? rp[i >> 1] : make_uint4(0u, 0u, 0u, 0u);
    if (sc == nullptr && rp == nullptr) {  // the accumulators as they are
      pk[2 * i] = act_pack2<ACT>(__uint_as_float(raw[4 * i]), __uint_as_float(raw[4 * i + 1]));
      pk[2 * i + 1] = act_pack2<ACT>(__uint_as_float(raw[4 * i + 2]), __uint_as_float(raw[4 * i + 3]));
      continue;
    }
    if (sc == nullptr) {
      float a = __uint_as_float(raw[4 * i]), b = __uint_as_float(raw[4 * i + 1]);
      float c = __uint_as_float(raw[4 * i + 2]), d = __uint_as_float(raw[4 * i + 3]);
      const uint32_t w0 = (i & 1) ? rv.z : rv.x, w1 = (i & 1) ? rv.w : rv.y;
      a += __uint_as_float(w0 << 16);
      b += __uint_as_float(w0 & 0xFFFF0000u);
      c += __uint_as_float(w1 << 16);
      d += __uint_as_float(w1 & 0xFFFF0000u);
      pk[2 * i] = act_pack2<ACT>(a, b);
      pk[2 * i + 1] = act_pack2<ACT>(c, d);
      continue;
    }
    const float4 s4 = reinterpret_cast<const float4*>(sc)[i];
    const float4 h4 = reinterpret_cast<const float4*>(sh)[i];
    float a, b, c, d;
    f2_split(ffma2(f2(__uint_as_float(raw[4 * i]), __uint_as_float(raw[4 * i + 1])), f2(s4.x, s4.y),
                   f2(h4.x, h4.y)),
             a, b);
    f2_split(ffma2(f2(__uint_as_float(raw[4 * i + 2]), __uint_as_float(raw[4 * i + 3])), f2(s4.z, s4.w),
                   f2(h4.z, h4.w)),
             c, d);
    if (RES && rp) {
      const uint32_t w0 = (i & 1) ? rv.z : rv.x, w1 = (i & 1) ? rv.w : rv.y;
      a += __uint_as_float(w0 << 16);
      b += __uint_as_float(w0 & 0xFFFF0000u);
      c += __uint_as_float(w1 << 16);
      d += __uint_as_float(w1 & 0xFFFF0000u);
    }
    pk[2 * i] = act_pack2<ACT>(a, b);
    pk[2 * i + 1] = act_pack2<ACT>(c, d);
  }
}

// Which of the 16 packed pairs' bf16 values are non-zero (any pattern but +-0):
// bit i for the low value of pair i (column 2 i), bit 16 + i for the high one
// (column 2 i + 1): one compare and one three-input logic operation per pair.
__device__ __forceinline__ uint32_t nz_mask32(const uint32_t (&pk)[16]) {
  const __nv_bfloat162 zero = __floats2bfloat162_rn(0.f, 0.f);
  uint32_t m = 0u;
#pragma unroll
  for (int i = 0; i < 16; ++i)
    m |= __hneu2_mask(*reinterpret_cast<const __nv_bfloat162*>(&pk[i]), zero) & (0x00010001u << i);
  return m;
}

// nz_mask32's bit order to column order (bit c = column c).
__device__ __forceinline__ uint32_t nz_unpermute(uint32_t m) {
  uint32_t e = m & 0xFFFFu, o = m >> 16;
#pragma unroll
  for (int s = 8; s > 0; s >>= 1) {
    const uint32_t k = s == 8 ? 0x00FF00FFu : s == 4 ? 0x0F0F0F0Fu : s == 2 ? 0x33333333u : 0x55555555u;
    e = (e | (e << s)) & k;
    o = (o | (o << s)) & k;
  }
  return e | (o << 1);
}

// Everything a producer thread needs to know about work unit u (tile u / ks,
// K range u % ks): pure arithmetic on the parameters, 32-bit throughout.
struct UnitGeo {
  int t, ks, kb0, kb1;
  TileGeo g;
  bool rvalid;
  int img, oh, ow;
  int cb, rr, ss;  // conv = 2: channel block and tap (row, column) of block kb0
  int iy0, ix0;    // conv = 2: input origin of the tile
};

__device__ __forceinline__ UnitGeo unit_geo(const Geo& p, int u, int KS, int kblocks, int nt, int BN,
                                            int BK, int r) {
  UnitGeo q;
  q.t = u / KS;
  q.ks = u - q.t * KS;
  q.kb0 = q.ks * kblocks / KS;
  q.kb1 = (q.ks + 1) * kblocks / KS;
  q.g = tile_geo(p, q.t, nt, BN);
  tile_row(p, q.g, r, q.rvalid, q.img, q.oh, q.ow);
  q.cb = q.rr = q.ss = 0;
  if (p.conv == 2) {
    const int cb_per_tap = p.Cp / BK;
    const int tap = q.kb0 / cb_per_tap;
    q.cb = q.kb0 - tap * cb_per_tap;
    q.rr = tap / p.kw;
    q.ss = tap - q.rr * p.kw;
  }
  q.iy0 = q.g.th0 * p.stride - p.pad;
  q.ix0 = q.g.tw0 * p.stride - p.pad;
  return q;
}

template <int I>
struct IntConst {
  static constexpr int value = I;
};

template <int BN, int BK, int LEAN, bool STEM>
__global__ void __launch_bounds__(Warps<LEAN, STEM>::kThreads, 1)
    igemm_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB,
                 const __grid_constant__ CUtensorMap tmY, const __grid_constant__ CUtensorMap tmA32,
                 const __grid_constant__ CUtensorMap tmB32, const IgemmArgs P) {
  using C = Cfg<BN, BK, STEM>;
  constexpr int kMaxAccCols = C::kMaxAccCols;
  using Wp = Warps<LEAN, STEM>;
  constexpr int kEpiThreads = Wp::kEpiThreads;
  constexpr int kMmaWarp = Wp::kMma;
  constexpr int kProd = Wp::kProd, kProdThreads = 32 * kProd;
  constexpr int kEpiWarp0 = Wp::kEpi0, kEpiThread0 = 32 * kEpiWarp0;
  // accumulators in tensor memory: tiles in flight between the MMAs and the epilogue
  constexpr int kAcc = LEAN && BN <= 128 ? 4 : 2;
  constexpr uint32_t kTmemCols = kAcc * C::kAccCols;
  const Geo p = make_geo(P);
  // lean kernels (LEAN 1: no residual, 2: a residual and N % 8 == 0): TMA
  // producers only (mode 0 or 2), no K split, bf16 output (the host launches
  // them only then); the general kernel has modes 0 and 1
  if (LEAN) __builtin_assume(p.conv != 1);
  else __builtin_assume(p.conv != 2);
  if (STEM) __builtin_assume(p.conv == 0);
  const EpiDev ep = P.ep;
  const int act = P.ep.act;
  const __nv_bfloat16* const residual = LEAN == 1 ? nullptr : P.ep.residual;
  const int y_f32 = LEAN ? 0 : P.y_f32;
  const int emit = P.emit;
  const long long wlim = P.wait_limit > 0 ? P.wait_limit : kWaitLimitCycles;
  const __nv_bfloat16* const xin = P.x;
  const uint32_t* const in_blk = P.in_blk;
  const int in_C32 = P.in_C32;
  const unsigned long long* const in_rowbm = P.in_rowbm;
  const int in_W64 = P.in_W64;
  uint32_t* const err = P.err;
  void* const yout = P.y;
  constexpr int S = C::kStages;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) &
                                             ~uintptr_t(1023));
  const uint32_t sbase = smem_u32(smem);
  const uint32_t sA = sbase + C::kAOff;
  const uint32_t sB = sbase + C::kBOff;
  const uint32_t sStg = sbase + C::kStgOff;
  const uint32_t bar_full = sbase + C::kBarOff;  // + 8*s
  const uint32_t bar_empty = bar_full + 8 * S;   // + 8*s
  const uint32_t bar_accf = bar_empty + 8 * S;   // + 8*b
  const uint32_t bar_acce = bar_accf + 32;       // + 8*b
  const uint32_t bar_drain = bar_acce + 32;      // after an abort: the MMAs issued so far are done
  const uint32_t bar_resb = bar_drain + 8;       // the resident B blocks have landed
  int* flags = reinterpret_cast<int*>(smem + C::kFlagOff);
  int* stage_last = flags;                // [S]: 1 = last stage of its tile
  volatile int* s_abort = flags + S;      // CTA-wide abort request
  volatile int* s_last = flags + S + 2;   // [2] split K: this unit finishes its tile
  int* s_issued = flags + S + 4;          // stages the producer filled (for the drain after an abort)
  uint32_t* s_tmem = reinterpret_cast<uint32_t*>(flags + S + 1);
  uint32_t* s_kbits = reinterpret_cast<uint32_t*>(smem + C::kKBitsOff);
  unsigned long long* s_tap = reinterpret_cast<unsigned long long*>(smem + C::kTapOff);
  float* s_scale = reinterpret_cast<float*>(smem + C::kScaleOff);
  float* s_shift = s_scale + (LEAN ? BN : 2 * BN);
  uint32_t* s_cnt = reinterpret_cast<uint32_t*>(smem + C::kCntOff);  // [4][BN]
  uint32_t* s_acc = reinterpret_cast<uint32_t*>(smem + C::kAccOff);  // [N] non-zeros per column
  unsigned long long* s_rowbm = reinterpret_cast<unsigned long long*>(smem + C::kRowOff);
  uint32_t* s_blk = reinterpret_cast<uint32_t*>(smem + C::kBlkOff);

  const int warp = threadIdx.x >> 5;
  const int lane = threadIdx.x & 31;
  const int kblocks = (p.Ktot + BK - 1) / BK;
  const int kgroups = (p.Ktot + 31) / 32;  // 32-column groups of K (compacted zero-skip GEMM)
  const int nt = (p.N + BN - 1) / BN;
  const int mtiles = p.conv == 2 ? ((p.Nimg + p.bn - 1) / p.bn) * p.th * p.tw : (p.M + kBM - 1) / kBM;
  const int tiles = mtiles * nt;
  // split K (gather mode only): work unit u = (tile u / KS, K range u % KS); KS consecutive units
  // (run by neighbouring CTAs at the same time) share one output tile
  const int KS = (!LEAN && P.ksplit > 1) ? P.ksplit : 1;
  const int units = tiles * KS;
  // Lean epilogue: with four accumulators the 4 warps of a TMEM lane quarter
  // take every 4th tile each; with two (192- and 256-wide tiles), and where the
  // CTA has one tile (up to two of more than 64 columns), they share a tile's
  // 32-column blocks.  ncw: warps that share a quarter of a tile.
  constexpr int kQw = Wp::kEpi / 4;  // epilogue warps per lane quarter
  const int ncw = kAcc == 2 || units <= (BN > 64 ? 2 : 1) * (int)gridDim.x ? kQw : 1;
  // every tile of the CTA has the same columns
  const bool fixed_cols = nt == 1 || (int)gridDim.x % nt == 0 || units <= (int)gridDim.x;
  // Column counts of all tiles a CTA handles are summed in shared memory and
  // flushed once (atomics on one address from every tile would serialise in L2);
  // a lean CTA's only tile adds its columns' counts directly (shorter code, which
  // it runs once: 128 x 64 values with K = 64 6.9 -> 6.4 us with the clear).
  const bool one_tile = LEAN && !STEM && units <= (int)gridDim.x;
  const bool acc_smem = emit && p.N <= kMaxAccCols && !one_tile;

  if (!LEAN && P.dense_only) {
    // launched next to the fused small-FC kernel, which handles the zero-skip
    // path: decide first, and leave before any set-up when it is not ours
    pdl_wait();
    if (decide_path(P.disp) == 2) {
      pdl_trigger();
      return;
    }
  }
  if (threadIdx.x == 0) {
    for (int s = 0; s < S; ++s) {
      mbar_init(bar_full + 8 * s, STEM ? (uint32_t)kProd : (!LEAN && p.conv == 1) ? 129u : 1u);
      mbar_init(bar_empty + 8 * s, 1u);
    }
    for (int b = 0; b < kAcc; ++b) {
      mbar_init(bar_accf + 8 * b, 1u);
      mbar_init(bar_acce + 8 * b, LEAN ? (uint32_t)(4 * ncw) : (uint32_t)kEpiThreads);
    }
    mbar_init(bar_drain, 1u);
    mbar_init(bar_resb, 1u);
    *s_abort = 0;
    fence_mbar_init();
    if (p.conv != 1 && !STEM) prefetch_tmap(&tmA);
    prefetch_tmap(&tmB);
    if (p.conv == 0 && BK == 64 && !STEM) {
      prefetch_tmap(&tmA32);
      prefetch_tmap(&tmB32);
    }
    if (!y_f32) prefetch_tmap(&tmY);
  }
  if (warp == kMmaWarp) tmem_alloc(smem_u32(s_tmem), kTmemCols);
  const bool epi_warp = warp >= kEpiWarp0 && (LEAN || warp < kMmaWarp);
  if (acc_smem && epi_warp)
    for (int c = threadIdx.x - kEpiThread0; c < p.N; c += kEpiThreads) s_acc[c] = 0u;
  if (!LEAN && epi_warp) {
    for (int i = threadIdx.x - kEpiThread0; i < kBM; i += kEpiThreads) s_rowbm[i] = 0ull;
    for (int i = threadIdx.x - kEpiThread0; i < BN / 32; i += kEpiThreads) s_blk[i] = 0u;
  }
  // The producers' first work unit is laid out before the grid dependency
  // wait: no memory is read, and under programmatic dependent launch this
  // overlaps the tail of the kernel before.
  UnitGeo ug{};
  if (warp < kProd && (!LEAN || p.conv == 2) && (int)blockIdx.x < units)
    ug = unit_geo(p, blockIdx.x, KS, kblocks, nt, BN, BK, threadIdx.x);
  TileGeo tg{};  // dense lean producer: the CTA's tile `lane`
  if (LEAN && !STEM && warp == 0) {
    const int ul = (int)blockIdx.x + lane * (int)gridDim.x;
    tg = tile_geo(p, ul < units ? ul : (int)blockIdx.x, nt, BN);
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *s_tmem;
  if constexpr (LEAN && !STEM) {
    if (warp == 1) prefetch_weights_l2(P.w, p.N, p.Ktot, lane);
  }
  pdl_wait();
  pdl_trigger();
  const int path = decide_path(P.disp);
  // with dense_only the zero-skip kernel of this launch runs instead
  const bool run = !(!LEAN && P.dense_only && path == 2);
  if (run) record_path(P.disp, path);
  // (nothing can be left out of the loads of a stem, a GEMM with one K block or
  // an input without block masks)
  const bool skip = !STEM && path == 2 && !(p.conv == 0 && (kblocks == 1 || in_blk == nullptr));
  // zero-skip GEMM with 64-wide K blocks: stages hold two occupied 32-column
  // groups each (compacted), loaded as 32-column boxes with the 64-byte swizzle
  const bool compact = skip && p.conv == 0;  // (kblocks > 1: BK = 64)

  // fixed columns and, on the dense path, a K range that fits the ring: its B
  // blocks are loaded once and stay, and the ring carries A alone (a 1x1 expansion
  // [32,112,112,16] -> 96 spent 11 of 53 us on reloading its 12 KB of weights per tile)
  const bool resident_b =
      STEM || (LEAN && !skip && fixed_cols && kblocks <= S && units > (int)gridDim.x);

  if (!run) {
    // nothing to do; fall through to the common exit (TMEM is freed there)
  } else if (warp < kProd) {
    // ------------------------------------------------------------------ producers
    if constexpr (STEM) {
      // The A tiles of a stem: K column kr * seg + e of pixel (n, oh, ow) is
      // element e of the kw * C window of input row oh * stride - pad + kr, which
      // is contiguous in NHWC.  A tile's input rows are staged by cp.async (the
      // next tile's while this one is built), as the 16-byte chunks that hold
      // them, so that row v starts at lead + (its misalignment); columns outside
      // the image are zeros around the data, rows outside are zero rows.  One
      // lane builds one pixel's window of one kernel row: words by a funnel
      // shift (a window may start on an odd element), 16-byte chunks out.  All
      // seven warps do both in turn: with the staging left to one warp the tile
      // waited for it (71 us against 62 on [32,224,224,3] 7x7/2).
      const StemGeo G = P.stem;
      const int tid = threadIdx.x;
      uint8_t* const rowbuf = smem + C::kStemOff;
      const int row_elems = G.W * G.C;
      const int wlen = G.kw * G.C, sc = G.stride * G.C, pad_c = G.pad * G.C;
      const int nseg = G.seg >> 3;
      const uint32_t xmis = (uint32_t)((reinterpret_cast<uintptr_t>(G.x) >> 1) & 7);  // elements past a 16-byte boundary
      if (warp == 0 && elect_one()) {
        mbar_arrive_expect_tx(bar_resb, (uint32_t)(kblocks * C::kBStage));
        for (int kb = 0; kb < kblocks; ++kb) tma_load_2d(sB + kb * C::kBStage, &tmB, bar_resb, kb * BK, 0);
      }
      // zeros everywhere: the margins stay, and the K columns past kh * seg
      for (int i = tid; i < 2 * kStemRowBytes / 16; i += kProdThreads)
        reinterpret_cast<uint4*>(rowbuf)[i] = make_uint4(0u, 0u, 0u, 0u);
      for (int i = tid; i < S * C::kAStage / 16; i += kProdThreads)
        reinterpret_cast<uint4*>(smem + C::kAOff)[i] = make_uint4(0u, 0u, 0u, 0u);
      named_bar_sync(1, kProdThreads);
      const int chunks = (row_elems + 14) >> 3;  // of a row, whatever its misalignment
      // requests the rows of tile u into buffer b (a warp a row) and writes its tables
      auto stage_rows = [&](int u, int b) {
        int* const s_row = reinterpret_cast<int*>(smem + C::kStemTabOff + b * C::kStemTab);  // window origin of row v
        uint32_t* const s_pix = reinterpret_cast<uint32_t*>(s_row + kMaxStemRows);
        const int m0 = u * kBM;
        const int m1 = m0 + kBM < p.M ? m0 + kBM : p.M;
        const int g0 = (int)__umulhi((uint32_t)m0, G.wo_mul) >> G.wo_shift, ow0 = m0 - g0 * G.Wo;  // m0 / Wo
        const int span = (int)(__umulhi((uint32_t)(ow0 + m1 - m0 - 1), G.wo_mul) >> G.wo_shift) + 1;  // output rows of the tile
        const int n0 = (int)__umulhi((uint32_t)g0, G.ho_mul) >> G.ho_shift, oh0 = g0 - n0 * G.Ho;
        const int ka = G.Ho - oh0 < span ? G.Ho - oh0 : span;  // ... of them in image n0
        const int rows_a = G.kh + (ka - 1) * G.stride;
        const int rows = rows_a + (span > ka ? G.kh + (span - ka - 1) * G.stride : 0);
        const uint32_t dst0 = smem_u32(rowbuf + b * kStemRowBytes);
        for (int v = warp; v < rows; v += kProd) {
          const bool second = v >= rows_a;
          const int ih = second ? v - rows_a - G.pad : oh0 * G.stride - G.pad + v;
          const bool live = ih >= 0 && ih < G.H;
          const int64_t e0 = ((int64_t)(n0 + (second ? 1 : 0)) * G.H + (live ? ih : 0)) * row_elems;  // element of x
          const int mis = (int)((uint32_t)e0 + xmis) & 7;
          const __nv_bfloat16* src = G.x + e0 - mis;
          const uint32_t dst = dst0 + (uint32_t)((v * G.pitch + G.lead) * 2);
          const int end = live ? mis + row_elems : 0;  // elements from the first chunk's start
          for (int c = lane; c < chunks; c += 32) {
            const int left = end - 8 * c;
            cp_async_16(dst + 16u * c, left > 0 ? src + 8 * c : src, left >= 8 ? 16u : left > 0 ? (uint32_t)(2 * left) : 0u);
          }
          if (lane == 0) s_row[v] = v * G.pitch + G.lead + (live ? mis : 0) - pad_c;
        }
        if (tid < kBM) {
          const int at = ow0 + (m0 + tid < m1 ? tid : m1 - 1 - m0);
          const int k = (int)__umulhi((uint32_t)at, G.wo_mul) >> G.wo_shift, ow = at - k * G.Wo;
          s_pix[tid] = ((uint32_t)(k < ka ? k * G.stride : rows_a + (k - ka) * G.stride) << 24) | (uint32_t)(ow * sc);
        }
      };
      // what a window's last chunk keeps of its four words
      uint32_t keep[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const int have = wlen - (8 * (nseg - 1) + 2 * i);
        keep[i] = have >= 2 ? 0xFFFFFFFFu : have == 1 ? 0xFFFFu : 0u;
      }
      int it = 0;
      bool ok = true;
      if ((int)blockIdx.x < units) stage_rows(blockIdx.x, 0);
      cp_async_commit();
      for (int u = blockIdx.x; u < units; u += gridDim.x, ++it) {
        const int b = it & 1, slot = it & 1;
        if (u + (int)gridDim.x < units) stage_rows(u + gridDim.x, b ^ 1);
        cp_async_commit();
        cp_async_wait<1>();
        named_bar_sync(1, kProdThreads);  // this tile's rows and tables are complete
        const int* const s_row = reinterpret_cast<const int*>(smem + C::kStemTabOff + b * C::kStemTab);
        const uint32_t* const s_pix = reinterpret_cast<const uint32_t*>(s_row + kMaxStemRows);
        if (G.ragged && G.pad > 0) {
          // the chunks brought in neighbours' columns besides the row: zeros in
          // the pad * C columns either side that windows read
          uint16_t* const rows16 = reinterpret_cast<uint16_t*>(rowbuf + b * kStemRowBytes);
          for (int v = warp; v < G.rows; v += kProd)
            for (int k = lane; k < 2 * pad_c; k += 32) {
              const int at = s_row[v] + (k < pad_c ? k : row_elems + k);  // (s_row: pad_c before the data)
              if (at >= v * G.pitch && at < (v + 1) * G.pitch) rows16[at] = 0;  // (rows this tile has not: anything)
            }
          named_bar_sync(1, kProdThreads);
        }
        if (it >= S)
          ok = ok && mbar_wait_warp(bar_empty + 8 * slot, (uint32_t)(((it >> 1) & 1) ^ 1), err, s_abort, kErrTimeoutEmpty, wlim);
        if (ok) {
          const uint32_t* const words = reinterpret_cast<const uint32_t*>(rowbuf + b * kStemRowBytes);
          const uint32_t a0 = sA + slot * C::kAStage;
          auto build = [&](auto nseg_c) {
            constexpr int NS = decltype(nseg_c)::value;
#pragma unroll 4
            for (int unit = warp; unit < 4 * G.kh; unit += kProd) {
              const int rr = (unit & 3) * 32 + lane, kr = unit >> 2;
              const uint32_t px = s_pix[rr];
              const int e = s_row[(px >> 24) + kr] + (int)(px & 0xFFFFFFu);
              const uint32_t* src = words + (e >> 1);
              const uint32_t sh = (uint32_t)(e & 1) * 16u;
              uint32_t w[4 * NS + 1];
#pragma unroll
              for (int i = 0; i <= 4 * NS; ++i) w[i] = src[i];
#pragma unroll
              for (int i = 0; i < 4 * NS; ++i) {
                w[i] = __funnelshift_r(w[i], w[i + 1], sh);
                if (i >= 4 * (NS - 1)) w[i] &= keep[i & 3];
              }
#pragma unroll
              for (int q = 0; q < NS; ++q) {
                const int kc = kr * NS + q;  // 16-byte chunk of the K axis
                sts_u4(a0 + (uint32_t)((kc >> 3) * (kBM * BK * 2)) + swz_offset<BK>(rr, kc & 7),
                       make_uint4(w[4 * q], w[4 * q + 1], w[4 * q + 2], w[4 * q + 3]));
              }
            }
          };
          if (nseg == 3) build(IntConst<3>{});
          else if (nseg == 2) build(IntConst<2>{});
          else build(IntConst<1>{});
          fence_proxy_async_smem();
          __syncwarp();
          if (lane == 0) mbar_arrive(bar_full + 8 * slot);
        }
        named_bar_sync(1, kProdThreads);  // buffer b and its tables are free for the tile after next
      }
      cp_async_wait<0>();
      if (tid == 0) *s_issued = 0;  // (no TMA copies into the ring)
    } else if (compact) {
      // Zero-skip GEMM: the converged warp walks the tile's 128-row block of the
      // input's masks, 32 column groups a step (one word a lane, the next step's
      // words loaded ahead, across tiles), and issues the occupied groups in
      // pairs (an aligned pair as one 64-wide K block).  A stage is held back until the next occupied group or the tile's
      // end is known, so that the last one can be marked; a tile with none runs
      // group 0 (all zero) so that its accumulator is written.
      if (warp == 0) {
        const bool el = elect_one();
        int it = 0, slot = 0;
        uint32_t ph = 0u;
        bool ok = true;
        auto issue = [&](int ga, int gb, int m0, int n0, bool last) {
          ok = ok && (it < S || mbar_wait_warp(bar_empty + 8 * slot, ph ^ 1u, err, s_abort, kErrTimeoutEmpty, wlim));
          if (!ok) return;
          if (el) {
            const uint32_t fb = bar_full + 8 * slot;
            const int nh = gb >= 0 ? 2 : 1;
            const bool whole = gb == ga + 1 && (ga & 1) == 0;  // a 64-wide K block: one box of 128-byte rows
            stage_last[slot] = (last ? 1 : 0) | (nh == 1 ? 2 : 0) | (whole ? 4 : 0);
            mbar_arrive_expect_tx(fb, (uint32_t)(nh * (kBM * 64 + BN * 64)));
            if (whole) {
              tma_load_2d(sA + slot * C::kAStage, &tmA, fb, ga * 32, m0);
              tma_load_2d(sB + slot * C::kBStage, &tmB, fb, ga * 32, n0);
            } else {
              tma_load_2d(sA + slot * C::kAStage, &tmA32, fb, ga * 32, m0);
              tma_load_2d(sB + slot * C::kBStage, &tmB32, fb, ga * 32, n0);
              if (nh == 2) {
                tma_load_2d(sA + slot * C::kAStage + kBM * 64, &tmA32, fb, gb * 32, m0);
                tma_load_2d(sB + slot * C::kBStage + BN * 64, &tmB32, fb, gb * 32, n0);
              }
            }
          }
          __syncwarp();
          ++it;
          if (++slot == S) {
            slot = 0;
            ph ^= 1u;
          }
        };
        auto word_at = [&](int u, int c) -> uint32_t {  // group 32 c + lane of tile u's block
          if (u >= units) return 0u;
          const int mi = nt == 1 ? u : u / nt;
          const int gi = c * 32 + lane;
          return gi < kgroups ? in_blk[(int64_t)mi * in_C32 + gi] : 0u;
        };
        const int steps = (kgroups + 31) / 32;
        uint32_t ahead = word_at(blockIdx.x, 0);
        for (int u = blockIdx.x; u < units && ok; u += gridDim.x) {
          const int mi = nt == 1 ? u : u / nt;
          const int m0 = mi * kBM, n0 = (u - mi * nt) * BN;
          int ga = -1, gb = -1;  // the stage held back
          for (int c = 0; c < steps; ++c) {
            uint32_t bits = __ballot_sync(0xffffffffu, ahead != 0u);
            ahead = c + 1 < steps ? word_at(u, c + 1) : word_at(u + (int)gridDim.x, 0);
            for (; bits; bits &= bits - 1u) {
              const int gi = c * 32 + __ffs(bits) - 1;
              if (ga < 0) {
                ga = gi;
              } else if (gb < 0) {
                gb = gi;
              } else {
                issue(ga, gb, m0, n0, false);
                ga = gi;
                gb = -1;
              }
            }
          }
          issue(ga < 0 ? 0 : ga, gb, m0, n0, true);
        }
        if (lane == 0) *s_issued = it;  // stages this CTA filled (TMA copies issued)
      }
    } else if (p.conv != 1 && !skip) {
      // Dense path (mode 2: lean kernels only): one converged warp, one elected lane issues.  The tiles'
      // origins (a few integer divisions each) are computed for 32 tiles at a
      // time, one per lane.
      if (warp == 0) {
        const bool el = elect_one();
        if (resident_b && el) {
          const int n0 = ((int)blockIdx.x % nt) * BN;
          mbar_arrive_expect_tx(bar_resb, (uint32_t)(kblocks * C::kBStage));
          for (int kb = 0; kb < kblocks; ++kb) tma_load_2d(sB + kb * C::kBStage, &tmB, bar_resb, kb * BK, n0);
        }
        const uint32_t bytes = resident_b ? (uint32_t)C::kAStage : (uint32_t)C::kStageBytes;
        const int cb_per_tap = p.Cp / BK;
        int it = 0, slot = 0;
        uint32_t ph = 0u;
        bool ok = true;
        for (int u0 = blockIdx.x; u0 < units && ok; u0 += 32 * (int)gridDim.x) {
          if (u0 != (int)blockIdx.x || !LEAN) {
            const int ul = u0 + lane * (int)gridDim.x;
            tg = tile_geo(p, ul < units ? ul : u0, nt, BN);
          }
          const TileGeo gl = tg;
          const int yl = p.conv == 2 ? gl.th0 * p.stride - p.pad : gl.m0, xl = gl.tw0 * p.stride - p.pad;
          for (int i = 0; i < 32 && u0 + i * (int)gridDim.x < units && ok; ++i) {
            const int y0 = __shfl_sync(0xffffffffu, yl, i), x0 = __shfl_sync(0xffffffffu, xl, i);
            const int b0 = __shfl_sync(0xffffffffu, gl.tn0, i), n0 = __shfl_sync(0xffffffffu, gl.n0, i);
            int cb = 0, rr = 0, ss = 0;  // conv = 2: channel block and tap of block kb
            for (int kb = 0; kb < kblocks; ++kb) {
              // (the ring's first lap, whose slots are free, waits for nothing)
              if (it >= S && !mbar_wait_warp(bar_empty + 8 * slot, ph ^ 1u, err, s_abort, kErrTimeoutEmpty, wlim)) {
                ok = false;
                break;
              }
              if (el) {
                const uint32_t fb = bar_full + 8 * slot;
                mbar_arrive_expect_tx(fb, bytes);
                if (p.conv == 0)
                  tma_load_2d(sA + slot * C::kAStage, &tmA, fb, kb * BK, y0);
                else
                  tma_load_4d(sA + slot * C::kAStage, &tmA, fb, cb * BK, x0 + ss, y0 + rr, b0);
                if (!resident_b) tma_load_2d(sB + slot * C::kBStage, &tmB, fb, kb * BK, n0);
              }
              __syncwarp();
              ++it;
              if (++slot == S) {
                slot = 0;
                ph ^= 1u;
              }
              if (p.conv == 2 && ++cb == cb_per_tap) {
                cb = 0;
                if (++ss == p.kw) {
                  ss = 0;
                  ++rr;
                }
              }
            }
          }
        }
        if (lane == 0) *s_issued = it;  // stages this CTA filled (TMA copies issued)
      }
    } else {
    // The gather of mode 1 (general kernel), or mode 2 on the zero-skip path (lean).
    const int r = threadIdx.x;
    int it = 0;        // stages filled so far (ring position)
    int pending = 0;   // mode 1: filled stages whose A arrivals are still owed
    bool ok = true;
    for (int u = blockIdx.x; u < units; u += gridDim.x) {
      if (u != (int)blockIdx.x) ug = unit_geo(p, u, KS, kblocks, nt, BN, BK, r);
      const int kb0 = ug.kb0, kb1 = ug.kb1;
      const TileGeo g = ug.g;
      const bool rvalid = ug.rvalid;
      const int img = ug.img, oh = ug.oh, ow = ug.ow;
      int last = kb1 - 1;
      if (skip) {
        // ---- occupied K blocks of this tile
        named_bar_sync(1, kProdThreads);  // thread 0 is done with the previous tile's bits
        if (r < kMaxTaps) s_tap[r] = 0ull;
        named_bar_sync(1, kProdThreads);
        const int taps = p.kh * p.kw < kMaxTaps ? p.kh * p.kw : kMaxTaps;
        auto mask_taps = [&](int t0, bool rv, int ri, int ry, int rx) {
          unsigned long long wv[8];
#pragma unroll
          for (int u = 0; u < 8; ++u) {  // issue 8 taps' loads before reducing any
            const int tp = t0 + u;
            const int ih = ry * p.stride - p.pad + tp / p.kw;
            const int iw = rx * p.stride - p.pad + tp % p.kw;
            wv[u] = 0ull;
            if (in_rowbm && tp < taps && rv && ih >= 0 && ih < p.H && iw >= 0 && iw < p.W)
              wv[u] = in_rowbm[(((int64_t)ri * p.H + ih) * p.W + iw) * in_W64];
          }
#pragma unroll
          for (int u = 0; u < 8; ++u) {
            unsigned long long w = wv[u];
#pragma unroll
            for (int s = 16; s > 0; s >>= 1) w |= __shfl_xor_sync(0xffffffffu, w, s);
            if (lane == 0 && w) atomicOr(&s_tap[t0 + u], w);
          }
        };
        if constexpr (LEAN) {
          // three warps share the four groups of 32 rows by 8 taps at a time
          for (int part = warp; part < 4 * ((taps + 7) / 8); part += kProd) {
            bool rv;
            int ri, ry, rx;
            tile_row(p, g, (part & 3) * 32 + lane, rv, ri, ry, rx);
            mask_taps((part >> 2) * 8, rv, ri, ry, rx);
          }
        } else {
          for (int t0 = 0; t0 < taps; t0 += 8) mask_taps(t0, rvalid, img, oh, ow);
        }
        named_bar_sync(1, kProdThreads);
        // no per-tap masks (too many taps, wide rows, or an input given without
        // row bitmaps): keep every block
        const bool many = p.kh * p.kw > kMaxTaps || in_W64 > 1 || in_rowbm == nullptr;
        for (int w0 = 0; w0 < kblocks && w0 < kMaxKWords * 32; w0 += kProdThreads) {
          const int kb = w0 + r;
          bool occ = false;
          if (kb < kblocks) {
            if (many) {
              occ = true;
            } else {
#pragma unroll
              for (int j = 0; j < BK / 8; ++j) {
                const int flat = kb * BK + 8 * j;
                if (flat >= p.Ktot) break;
                const int tp = flat / p.Cp;
                const int c = flat - tp * p.Cp;
                occ |= ((s_tap[tp] >> (c >> 6)) & 1ull) != 0ull;
              }
            }
          }
          const uint32_t bits = __ballot_sync(0xffffffffu, occ);
          if (lane == 0 && (w0 >> 5) + warp < kMaxKWords) s_kbits[(w0 >> 5) + warp] = bits;
        }
        named_bar_sync(1, kProdThreads);
        // last occupied block of this unit's K range; a range with none still
        // runs its first block (whose data is all zero)
        last = kb0;
        for (int kb = kb1 - 1; kb > kb0; --kb) {
          if (kb >= kMaxKWords * 32 || ((s_kbits[kb >> 5] >> (kb & 31)) & 1u)) {
            last = kb;
            break;
          }
        }
      }
      if (!ok) continue;  // keep the skip-mask barriers in step; issue nothing more
      if constexpr (LEAN) {
        if (r == 0) {
          // Ring slot, phase and the (tap, channel block) of each K block advance
          // incrementally, with no divisions in the loop, and the ring's first lap
          // (whose slots are free by construction) waits for nothing.
          const int cb_per_tap = p.Cp / BK;
          int slot = it % S;
          uint32_t ph = (uint32_t)((it / S) & 1);
          int cb = ug.cb, rr = ug.rr, ss = ug.ss;  // channel block and tap of block kb
          const int iy0 = ug.iy0, ix0 = ug.ix0;
          const uint32_t fb0 = bar_full, eb0 = bar_empty;
          for (int kb = kb0; kb <= last; ++kb) {
            if (kb == last || kb >= kMaxKWords * 32 || ((s_kbits[kb >> 5] >> (kb & 31)) & 1u)) {
              if (it >= S && !mbar_wait(eb0 + 8 * slot, ph ^ 1u, err, s_abort, kErrTimeoutEmpty, wlim)) {
                ok = false;
                break;
              }
              const uint32_t fb = fb0 + 8 * slot;
              stage_last[slot] = (kb == last) ? 1 : 0;
              mbar_arrive_expect_tx(fb, (uint32_t)C::kStageBytes);
              tma_load_4d(sA + slot * C::kAStage, &tmA, fb, cb * BK, ix0 + ss, iy0 + rr, g.tn0);
              tma_load_2d(sB + slot * C::kBStage, &tmB, fb, kb * BK, g.n0);
              ++it;
              if (++slot == S) {
                slot = 0;
                ph ^= 1u;
              }
            }
            if (++cb == cb_per_tap) {
              cb = 0;
              if (++ss == p.kw) {
                ss = 0;
                ++rr;
              }
            }
          }
        }
      } else {
        // Implicit-GEMM gather: row r is output pixel m0 + r.
        const int ih0 = oh * p.stride - p.pad;
        const int iw0 = ow * p.stride - p.pad;
        const __nv_bfloat16* ximg = xin + (int64_t)img * p.H * p.W * p.Cp;
        for (int kb = kb0; kb <= last; ++kb) {
          if (skip && kb != last && kb < kMaxKWords * 32 && !((s_kbits[kb >> 5] >> (kb & 31)) & 1u))
            continue;
          const int slot = it % S;
          const uint32_t ph = (uint32_t)((it / S) & 1);
          if (!mbar_wait(bar_empty + 8 * slot, ph ^ 1u, err, s_abort, kErrTimeoutEmpty, wlim)) {
            ok = false;
            break;
          }
          if (r == 0) {
            stage_last[slot] = (kb == last) ? 1 : 0;
            mbar_arrive_expect_tx(bar_full + 8 * slot, (uint32_t)C::kBStage);
            tma_load_2d(sB + slot * C::kBStage, &tmB, bar_full + 8 * slot, kb * BK, g.n0);
          }
          const uint32_t dst = sA + slot * C::kAStage;
          // (tap, channel) of the block's first 8-channel chunk by division,
          // the block's other chunks by stepping (C % 8 == 0)
          const int flat0 = kb * BK;
          const int tp0 = flat0 / p.Cp;
          int c = flat0 - tp0 * p.Cp;
          int rr = tp0 / p.kw;
          int ss = tp0 - rr * p.kw;
#pragma unroll
          for (int j = 0; j < BK / 8; ++j) {
            const int flat = flat0 + 8 * j;
            const int ih = ih0 + rr, iw = iw0 + ss;
            const bool val = rvalid && flat < p.Ktot && ih >= 0 && ih < p.H && iw >= 0 && iw < p.W;
            const __nv_bfloat16* src = val ? ximg + ((int64_t)ih * p.W + iw) * p.Cp + c : xin;
            cp_async_16(dst + swz_offset<BK>(r, j), src, val ? 16u : 0u);
            c += 8;
            if (c == p.Cp) {
              c = 0;
              if (++ss == p.kw) {
                ss = 0;
                ++rr;
              }
            }
          }
          cp_async_commit();
          ++it;
          ++pending;
          if (pending > C::kLag) {
            cp_async_wait<C::kLag>();
            fence_proxy_async_smem();
            mbar_arrive(bar_full + 8 * ((it - 1 - C::kLag) % S));
            --pending;
          }
        }
      }
    }
    if (r == 0) *s_issued = it;  // stages this CTA filled (TMA copies issued)
    if (!LEAN) {
      cp_async_wait<0>();
      fence_proxy_async_smem();
      for (int q = pending; q > 0; --q) mbar_arrive(bar_full + 8 * ((it - q) % S));
    }
    }
  } else if (warp == kMmaWarp) {
    // ------------------------------------------------------------------ MMA issue
    // The warp stays converged; `el` (one lane) issues.  The ring position is
    // carried as descriptors and barrier addresses, so a stage costs a wait, a
    // few uniform additions, its MMAs and a commit.
    constexpr uint32_t idesc = idesc_bf16_f32(kBM, BN);
    const bool el = elect_one();
    const uint64_t ad0 = smem_desc_kmajor<BK>(sA), bd0 = smem_desc_kmajor<BK>(sB);
    uint64_t ad = ad0, bd = bd0;
    int slot = 0, j = 0;
    uint32_t ph = 0;
    auto next = [&]() {
      ad += C::kAStage / 16;
      bd += C::kBStage / 16;
      if (++slot == S) {
        slot = 0;
        ph ^= 1u;
        ad = ad0;
        bd = bd0;
      }
    };
    // One dense stage.  k-steps advance the start-address field by 32 B (2
    // units); the accumulate flag is a constant of each MMA (a flag computed
    // at run time roughly halves the issue rate).
    auto stage = [&](uint32_t d, uint64_t b0, auto first) -> bool {
      if (!mbar_wait_warp(bar_full + 8 * slot, ph, err, s_abort, kErrTimeoutFull, wlim)) return false;
      tc_fence_after();
      if (el) {
        tc_mma_bf16(d, ad, b0, idesc, decltype(first)::value ? 0u : 1u);
#pragma unroll
        for (int k = 1; k < BK / 16; ++k) tc_mma_bf16(d, ad + (uint64_t)(2 * k), b0 + (uint64_t)(2 * k), idesc, 1u);
        tc_commit(bar_empty + 8 * slot);
      }
      __syncwarp();
      next();
      return true;
    };
    const bool halves = !STEM && BK == 64 && path == 2 && p.conv == 0 && kblocks == 1 && kgroups == 2 && in_blk != nullptr;
    uint32_t half_bits = 0u;  // lane l: the occupied groups of the CTA's tile j + l
    bool ok = !resident_b || mbar_wait_warp(bar_resb, 0u, err, s_abort, kErrTimeoutFull, wlim);
    if (resident_b) tc_fence_after();
    for (int u = blockIdx.x; u < units && ok; u += gridDim.x, ++j) {
      const int b = j & (kAcc - 1);
      if (!mbar_wait_warp(bar_acce + 8 * b, (uint32_t)(((j / kAcc) & 1) ^ 1), err, s_abort, kErrTimeoutAcc, wlim))
        break;
      tc_fence_after();
      const uint32_t d = tmem + (uint32_t)b * C::kAccCols;
      if constexpr (STEM) {
        // the whole A tile is one stage; its k-steps alternate between two halves
        // of the accumulator (the epilogue adds them): each sum is rounded half as
        // often.  The 7x7's eleven k-steps in one accumulator left 4 % more error
        // than the ten of im2col rows ([8,224,224,3] to 64, of the bf16 result:
        // 2.66e-5, 2.78e-5 and, this way, 2.01e-5 for 1.4 us of 43).
        const int nks = (p.Ktot + 15) / 16;
        ok = mbar_wait_warp(bar_full + 8 * slot, ph, err, s_abort, kErrTimeoutFull, wlim);
        if (ok) {
          tc_fence_after();
          if (el) {
#pragma unroll
            for (int k = 0; k < 12; ++k)
              if (k < nks)
                tc_mma_bf16(d + (uint32_t)(k & 1) * 64u, ad + (uint64_t)((k >> 2) * (kBM * BK * 2 / 16) + 2 * (k & 3)),
                            bd0 + (uint64_t)((k >> 2) * (C::kBStage / 16) + 2 * (k & 3)), idesc, k < 2 ? 0u : 1u);
            tc_commit(bar_empty + 8 * slot);
          }
          __syncwarp();
          next();
        }
      } else if (halves) {
        // the zero-skip path of one K block of two groups: only the occupied one
        // (group 0 where the tile has none, so that its accumulator is written)
        if ((j & 31) == 0) {
          const int ul = u + lane * (int)gridDim.x;
          half_bits = 0u;
          if (ul < units) {
            const uint32_t* words = in_blk + (int64_t)(ul / nt) * in_C32;
            half_bits = (words[0] ? 1u : 0u) | (words[1] ? 2u : 0u);
          }
        }
        const uint32_t hv = __shfl_sync(0xffffffffu, half_bits, j & 31);
        ok = mbar_wait_warp(bar_full + 8 * slot, ph, err, s_abort, kErrTimeoutFull, wlim);
        if (ok) {
          tc_fence_after();
          const uint64_t b0 = resident_b ? bd0 : bd;
          if (el) {
            if (hv != 2u) {
              tc_mma_bf16(d, ad, b0, idesc, 0u);
              tc_mma_bf16(d, ad + 2, b0 + 2, idesc, 1u);
            }
            if (hv & 2u) {
              if (hv == 3u) tc_mma_bf16(d, ad + 4, b0 + 4, idesc, 1u);
              else tc_mma_bf16(d, ad + 4, b0 + 4, idesc, 0u);
              tc_mma_bf16(d, ad + 6, b0 + 6, idesc, 1u);
            }
            tc_commit(bar_empty + 8 * slot);
          }
          __syncwarp();
          next();
        }
      } else if (!skip) {
        // every K block of the unit
        const int ks = KS == 1 ? 0 : u - (u / KS) * KS;
        const int n = KS == 1 ? kblocks : (ks + 1) * kblocks / KS - ks * kblocks / KS;
        ok = stage(d, resident_b ? bd0 : bd, BoolConst<true>{});
        for (int i = 1; i < n && ok; ++i)
          ok = stage(d, resident_b ? bd0 + (uint64_t)(i * (C::kBStage / 16)) : bd, BoolConst<false>{});
      } else {
        // the occupied ones: the producer marks a unit's last stage (bit 0)
        bool first = true, last = false;
        while (!last) {
          if (!mbar_wait_warp(bar_full + 8 * slot, ph, err, s_abort, kErrTimeoutFull, wlim)) {
            ok = false;
            break;
          }
          tc_fence_after();
          const int sflags = stage_last[slot];
          last = (sflags & 1) != 0;
          if (el) {
            if (compact && !(sflags & 4)) {
              // one or two 32-column groups, each 128 (A) / BN (B) rows of 64
              // bytes with the 64-byte swizzle: two k-steps of 16 per group
              const uint32_t a = sA + slot * C::kAStage, bb = sB + slot * C::kBStage;
              const uint64_t a0 = smem_desc_sw64(a), b0 = smem_desc_sw64(bb);
              if (first) tc_mma_bf16(d, a0, b0, idesc, 0u);
              else tc_mma_bf16(d, a0, b0, idesc, 1u);
              tc_mma_bf16(d, a0 + 2, b0 + 2, idesc, 1u);
              if (!(sflags & 2)) {
                const uint64_t a1 = smem_desc_sw64(a + kBM * 64), b1 = smem_desc_sw64(bb + BN * 64);
                tc_mma_bf16(d, a1, b1, idesc, 1u);
                tc_mma_bf16(d, a1 + 2, b1 + 2, idesc, 1u);
              }
            } else {
              if (first) tc_mma_bf16(d, ad, bd, idesc, 0u);
              else tc_mma_bf16(d, ad, bd, idesc, 1u);
#pragma unroll
              for (int k = 1; k < BK / 16; ++k)
                tc_mma_bf16(d, ad + (uint64_t)(2 * k), bd + (uint64_t)(2 * k), idesc, 1u);
            }
            tc_commit(bar_empty + 8 * slot);
          }
          __syncwarp();
          first = false;
          next();
        }
      }
      // (the fault injection of the error-path tests leaves the first
      // accumulator unsignalled: the epilogue's bounded wait runs out)
      if (ok && el && !(P.fault == kFaultSkipFirstAccCommit && j == 0)) tc_commit(bar_accf + 8 * b);
      __syncwarp();
    }
  } else if constexpr (LEAN) {
    // ------------------------------------------------------------- lean epilogue
    // The general epilogue's blocks (32 rows of one TMEM lane quarter x 32
    // columns, staged with the 64-byte swizzle, one TMA store each) without
    // K split or fp32 output.  No barrier inside the tile loop: a warp waits
    // for its tile's accumulator alone and writes its rows' bitmap words and
    // its block-column words itself; column counts go straight into the CTA's
    // column sums.  (With a barrier per tile the warps ran in lockstep, one
    // block's latency, about 3400 cycles, per tile and round: 16 warps were no
    // faster than 8.)
    const int q = warp & 3;
    const int r = q * 32 + lane;
    const int lane_col = lane < 16 ? 2 * lane : 2 * lane - 31;  // column of bit `lane` in nz_mask32's order
    const int ew = warp - kEpiWarp0;
    const int slots = ncw == 1 ? kQw : 1;            // tiles in work at a time
    const int slot = ncw == 1 ? ew >> 2 : 0;
    const int cw = ncw == 1 ? 0 : ew >> 2;           // this warp's 32-column blocks: cw, cw + ncw, ...
    int sw_ = 0, sh_ = 0, sn_ = 0;
    if (p.conv == 2) {
      const int rho = q * 32;
      sw_ = rho % p.bw;
      sh_ = (rho / p.bw) % p.bh;
      sn_ = rho / (p.bw * p.bh);
    }
    const uint32_t stg = sStg + (uint32_t)(ew * kWarpStgBytes);
    const bool affine = ep.bias != nullptr || ep.bn != nullptr;  // else the column affine is 1, 0
    // The column affine: one table when every tile of the CTA has the same
    // columns, else each warp computes a block's 32 columns ahead of it.
    float* const own = s_scale + 2 * BN + ew * 64;  // this warp's block: scale[32], shift[32]
    if (affine && fixed_cols) {
      const int n0 = ((int)blockIdx.x % nt) * BN;
      for (int c = threadIdx.x - kEpiThread0; c < BN; c += kEpiThreads) {
        float sc = 1.f, sh = 0.f;
        if (n0 + c < p.N) epi_affine(ep, p.N, n0 + c, sc, sh);
        s_scale[c] = sc;
        s_shift[c] = sh;
      }
      named_bar_sync(2, kEpiThreads);
    }
    const OccDev o = P.out_occ;
    // Column counts.  Up to 128-wide tiles (many small tiles per CTA): this
    // warp's blocks cw, cw + ncw, ... are added bit-sliced, seven tiles in three
    // planes in shared memory, before the planes are transposed.  Wider tiles:
    // every block's bits are transposed.
    constexpr bool kSliced = BN <= 128;
    constexpr int kBpw = BN / 32;
    uint32_t* const splane = reinterpret_cast<uint32_t*>(smem + C::kPlaneOff) + ew * (kBpw * 3 * 32) + lane;
    if (kSliced && emit && !one_tile)
#pragma unroll
      for (int i = 0; i < kBpw * 3; ++i) splane[i * 32] = 0u;
    int nsum = 0, n0_last = 0;
    uint32_t pend_bits = 0u;  // block-column words on their way out
    int pend_at = 0, npend = 0;
    auto flush_words = [&]() {
      if (lane < npend && pend_bits) atomicOr(&o.blk_mask[pend_at], nz_unpermute(pend_bits));
      npend = 0;
    };
    auto flush_counts = [&](uint32_t (&pl)[3], int ncol0) {
      // this lane's column (bit `lane` in nz_mask32's order): non-zeros in the warp's rows
      uint32_t cnt = __popc(warp_transpose32(pl[0]));
      if (kSliced && __any_sync(0xffffffffu, (pl[1] | pl[2]) != 0u))
        cnt += 2u * __popc(warp_transpose32(pl[1])) + 4u * __popc(warp_transpose32(pl[2]));
      pl[0] = pl[1] = pl[2] = 0u;
      const int col = ncol0 + lane_col;
      if (acc_smem) {
        if (cnt) atomicAdd(&s_acc[col], cnt);
      } else {
        if (cnt) atomicAdd(&o.col_nnz[col], cnt);  // (columns past N have none)
        const uint32_t sum = __reduce_add_sync(0xffffffffu, cnt);
        if (lane == 0 && sum) {
          atomicAdd(&o.tile_nnz[ncol0 >> 6], sum);
          atomicAdd(o.nnz, (unsigned long long)sum);
        }
      }
    };
    for (int j = slot;; j += slots) {
      const int u = (int)blockIdx.x + j * (int)gridDim.x;
      if (u >= units) break;
      const int b = j & (kAcc - 1);
      const TileGeo g = tile_geo(p, u, nt, BN);
      bool mvalid;
      int img, oh, ow;
      const int64_t m = tile_row(p, g, r, mvalid, img, oh, ow);
      const int ncb = p.N - g.n0 >= BN ? BN / 32 : (p.N - g.n0 + 31) >> 5;  // 32-column blocks of the tile
      if (LEAN == 2 && mvalid) {
        // this row's residual segments into L1 while the accumulator is pending
        const __nv_bfloat16* rrow = residual + m * p.N + g.n0;
        for (int c = cw; c < ncb; c += ncw) prefetch_l1(rrow + c * 32);
      }
      float nsc = 1.f, nsh = 0.f;  // the next block's affine of column `lane`
      auto load_affine = [&](int cblk) {
        const int c = g.n0 + cblk * 32 + lane;
        if (cblk < ncb && c < p.N) epi_affine(ep, p.N, c, nsc, nsh);
      };
      if (affine && !fixed_cols) load_affine(cw);
      const int blk = mvalid ? (int)(m >> 7) : -1;
      const uint32_t grp = p.conv == 2 ? __match_any_sync(0xffffffffu, blk) : 0xffffffffu;
      const bool leader = (__ffs(grp) - 1) == lane;
      if (!mbar_wait_warp(bar_accf + 8 * b, (uint32_t)((j / kAcc) & 1), err, s_abort, kErrTimeoutAcc, wlim)) break;
      tc_fence_after();
      const uint32_t tbase = tmem + ((uint32_t)(q * 32) << 16) + (uint32_t)b * C::kAccCols;
      unsigned long long tl = 0ull;  // this row's occupied 64-column tiles
      // One block: columns cblk * 32.. of the tile, accumulator values in raw;
      // the TMA store and this block's share of the output occupancy.
      auto block = [&](const uint32_t (&raw)[32], int cblk, uint32_t (&plane)[3]) {
        const int ncol0 = g.n0 + cblk * 32;
        const float* scg = !affine ? nullptr : fixed_cols ? s_scale + cblk * 32 : own;
        const float* shg = fixed_cols ? s_shift + cblk * 32 : own + 32;
        const uint4* rp =
            residual && mvalid ? reinterpret_cast<const uint4*>(residual + m * p.N + ncol0) : nullptr;
        const int rvalid = p.N - ncol0 < 32 ? p.N - ncol0 : 32;
        uint32_t pk[16];
        constexpr bool kRes = LEAN == 2;
        if (act == 1) affine_act_pack32<1, kRes>(raw, scg, shg, rp, rvalid, pk);
        else if (act == 2) affine_act_pack32<2, kRes>(raw, scg, shg, rp, rvalid, pk);
        else if (act == 0) affine_act_pack32<0, kRes>(raw, scg, shg, rp, rvalid, pk);
        else affine_act_pack32<3, kRes>(raw, scg, shg, rp, rvalid, pk);
        const uint32_t row_addr = stg + (uint32_t)lane * 64u;
        const int sx = (lane >> 1) & 3;
#pragma unroll
        for (int k = 0; k < 4; ++k)
          sts_u4(row_addr + (uint32_t)((k ^ sx) << 4), make_uint4(pk[4 * k], pk[4 * k + 1], pk[4 * k + 2], pk[4 * k + 3]));
        fence_proxy_async_smem();
        __syncwarp();
        if (lane == 0) {
          if (p.conv == 2)
            tma_store_4d(&tmY, stg, ncol0, g.tw0 + sw_, g.th0 + sh_, g.tn0 + sn_);
          else
            tma_store_2d(&tmY, stg, ncol0, g.m0 + q * 32);
          bulk_commit();
        }
        if (emit) {
          // row r's non-zero bits, in nz_mask32's order
          uint32_t rw = nz_mask32(pk);
          if (!mvalid) rw = 0u;
          else if (rvalid < 32) rw &= ((1u << (rvalid >> 1)) - 1u) * 0x00010001u;
          if (rw) tl |= 1ull << ((ncol0 >> 6) & 63);
          const uint32_t bits = __reduce_or_sync(grp, rw);
          const int word = ncol0 >> 5;
          if (p.conv == 2) {
            if (leader && blk >= 0 && bits && word < o.C32)
              atomicOr(&o.blk_mask[(int64_t)blk * o.C32 + word], nz_unpermute(bits));
          } else {
            // the tile is the whole block: its words wait, one per lane, and
            // leave 32 at a time
            if (lane == npend) {
              pend_bits = bits;
              pend_at = (g.m0 >> 7) * o.C32 + word;
            }
            if (++npend == 32) flush_words();
          }
          const uint32_t k1 = plane[0] & rw;
          plane[0] ^= rw;
          const uint32_t k2 = plane[1] & k1;
          plane[1] ^= k1;
          plane[2] |= k2;
        }
      };
      // (Two blocks per step, both accumulator loads in flight first, made
      // the kernel spill and was slower.)
#pragma unroll 1
      for (int cblk = cw; cblk < ncb; cblk += ncw) {
        uint32_t raw[32];
        tmem_ld32_nowait(tbase + (uint32_t)(cblk * 32), raw);
        if (affine && !fixed_cols) {
          own[lane] = nsc;
          own[32 + lane] = nsh;
          load_affine(cblk + ncw);
        }
        if (lane == 0) bulk_wait_read<0>();  // the last store from this buffer has read it
        __syncwarp();
        tmem_wait_ld32(raw);
        if (STEM && p.Ktot > 16) {  // the odd k-steps' half
          uint32_t odd[32];
          tmem_ld32_nowait(tbase + 64u + (uint32_t)(cblk * 32), odd);
          tmem_wait_ld32(odd);
#pragma unroll
          for (int i = 0; i < 32; ++i) raw[i] = __float_as_uint(__uint_as_float(raw[i]) + __uint_as_float(odd[i]));
        }
        if (cblk + ncw >= ncb) {  // accumulator b is free for the MMAs of tile j + kAcc
          tc_fence_before();
          __syncwarp();
          if (lane == 0) mbar_arrive(bar_acce + 8 * b);
        }
        uint32_t* const sp = splane + (ncw == 1 ? cblk : 0) * 96;
        uint32_t pl[3] = {0u, 0u, 0u};
        if (kSliced && emit && !one_tile)
#pragma unroll
          for (int i = 0; i < 3; ++i) pl[i] = sp[i * 32];
        block(raw, cblk, pl);
        if (emit && (!kSliced || !fixed_cols || one_tile || nsum == 6)) flush_counts(pl, g.n0 + cblk * 32);
        if (kSliced && emit && !one_tile)
#pragma unroll
          for (int i = 0; i < 3; ++i) sp[i * 32] = pl[i];
      }
      if (++nsum == 7) nsum = 0;
      n0_last = g.n0;
      if (cw >= ncb && lane == 0) mbar_arrive(bar_acce + 8 * b);  // no block of this tile
      if (emit && mvalid) {
        unsigned long long* dst = &o.row_bm[m * o.W64 + (g.n0 >> 12)];
        if (nt == 1 && ncw == 1) *dst = tl;  // all columns of the row's bitmap word
        else if (tl) atomicOr(dst, tl);
      }
    }
    if (emit) {
      flush_words();
      if (kSliced && fixed_cols && !one_tile)
        for (int k = 0; k < (ncw == 1 ? kBpw : 1); ++k) {
          uint32_t pl[3];
#pragma unroll
          for (int i = 0; i < 3; ++i) pl[i] = splane[k * 96 + i * 32];
          flush_counts(pl, n0_last + (cw + k * ncw) * 32);
        }
    }
    if (acc_smem) {
      named_bar_sync(2, kEpiThreads);
      unsigned long long total = 0ull;
      for (int c0 = 0; c0 < p.N; c0 += kEpiThreads) {
        const int c = c0 + (int)threadIdx.x - kEpiThread0;
        const uint32_t cnt = c < p.N ? s_acc[c] : 0u;
        if (cnt) atomicAdd(&o.col_nnz[c], cnt);
        uint32_t sum = cnt;
#pragma unroll
        for (int s = 16; s > 0; s >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, s);
        total += sum;
        if (lane == 0 && sum) atomicAdd(&o.tile_nnz[c >> 6], sum);
      }
      if (lane == 0 && total) atomicAdd(o.nnz, total);
    }
    if (lane == 0) bulk_wait_all();
  } else {
    // ------------------------------------------------------------------ epilogue
    // Each epilogue warp owns a 32-row x 32-column block of every 64-column
    // group (rows from its TMEM lane quarter, columns from its half) and
    // stores it on its own: staging in shared memory with the 64-byte swizzle
    // and one TMA store per block, so the warps never wait for each other
    // inside a tile.  The only barrier per tile publishes the column affine
    // (double-buffered by accumulator), plus one for the output occupancy.
    const int q = warp & 3;            // TMEM lane quarter of this warp
    const int hf = (warp - 4) >> 2;    // which 32 columns of each 64-column group
    const int ew = warp - 4;           // epilogue warp index
    const int r = q * 32 + lane;       // tile row
    const int et = threadIdx.x - kEpiThread0;  // 0..kEpiThreads-1
    const bool vec = (p.N % 8) == 0;
    const bool affine = ep.bias != nullptr || ep.bn != nullptr;  // else the column affine is 1, 0
    const uint32_t stg_base = sStg + (uint32_t)(ew * 2 * kWarpStgBytes);
    // Tile t covers columns (t % nt) BN..; when every tile of this CTA has the
    // same columns (one column tile, or a grid that is a multiple of the column
    // tiles) the column affine is computed once, into buffer 0, instead of per
    // tile (its global loads would otherwise sit on every tile's critical path)
    const bool same_cols = KS == 1 && fixed_cols;
    if (same_cols && (int)blockIdx.x < units) {
      const int n0 = ((int)blockIdx.x % nt) * BN;
      for (int c = et; c < BN; c += kEpiThreads) {
        float sc = 1.f, sh = 0.f;
        if (n0 + c < p.N) epi_affine(ep, p.N, n0 + c, sc, sh);
        s_scale[c] = sc;
        s_shift[c] = sh;
      }
    }
    int j = 0;
    int stg_count = 0;  // blocks this warp handed to TMA so far
    for (int u = blockIdx.x; u < units; u += gridDim.x, ++j) {
      const int t = u / KS, ks = u - (u / KS) * KS;
      const int b = j & 1;
      const TileGeo g = tile_geo(p, t, nt, BN);
      bool mvalid;
      int img, oh, ow;
      const int64_t m = tile_row(p, g, r, mvalid, img, oh, ow);
      float* const scb = s_scale + (same_cols ? 0 : b * BN);
      float* const shb = s_shift + (same_cols ? 0 : b * BN);
      // column affine of this tile into buffer b (its readers of tile j - 2
      // passed tile j - 1's barrier before any thread gets here)
      if (!same_cols) {
        for (int c = et; c < BN; c += kEpiThreads) {
          float sc = 1.f, sh = 0.f;
          if (g.n0 + c < p.N) epi_affine(ep, p.N, g.n0 + c, sc, sh);
          scb[c] = sc;
          shb[c] = sh;
        }
      }
      const bool ok = mbar_wait(bar_accf + 8 * b, (uint32_t)((j >> 1) & 1), err, s_abort, kErrTimeoutAcc, wlim);
      // publishes the affine, and makes the abort decision the same for every
      // epilogue warp (a warp that left alone would strand the others at a barrier)
      if (named_bar_or(2, kEpiThreads, !ok)) break;
      tc_fence_after();
      const uint32_t tbase = tmem + ((uint32_t)(q * 32) << 16) + (uint32_t)b * C::kAccCols;
      // split K: every unit stores its fp32 partial tile, then takes a ticket;
      // the unit that arrives last adds the others' partials and finishes the
      // tile (nobody waits for anybody)
      float* const ws_tile = KS > 1 ? P.ws + (int64_t)t * KS * kBM * BN : nullptr;
      if (KS > 1) {
        float* const mine = ws_tile + ((int64_t)ks * kBM + r) * BN + hf * 32;
#pragma unroll 1
        for (int gcol = 0; gcol < BN / 64; ++gcol) {
          uint32_t raw[32];
          tmem_ld32_nowait(tbase + (uint32_t)(gcol * 64 + hf * 32), raw);
          tmem_wait_ld32(raw);
          float4* dst = reinterpret_cast<float4*>(mine + gcol * 64);
#pragma unroll
          for (int i = 0; i < 8; ++i)
            __stcg(dst + i, make_float4(__uint_as_float(raw[4 * i]), __uint_as_float(raw[4 * i + 1]),
                                        __uint_as_float(raw[4 * i + 2]), __uint_as_float(raw[4 * i + 3])));
        }
        // One thread publishes the partial and takes the ticket: the barrier
        // orders every epilogue thread's stores before that thread's fence
        // (fences are cumulative), and the last arriver's fence after the
        // ticket orders the other units' partials before the reads below,
        // which the second barrier hands on to every thread.
        named_bar_sync(2, kEpiThreads);
        if (et == 0) {
          __threadfence();
          const int lst = atomicAdd(&P.ws_cnt[t], 1u) == (unsigned)(KS - 1) ? 1 : 0;
          if (lst) {
            __threadfence();
            P.ws_cnt[t] = 0u;  // every unit of the tile has arrived: ready for reuse
          }
          s_last[b] = lst;
        }
        named_bar_sync(2, kEpiThreads);
        if (!s_last[b]) {
          tc_fence_before();
          mbar_arrive(bar_acce + 8 * b);  // this unit's share is in the partial
          continue;
        }
      }
      const OccDev o = P.out_occ;  // registers, not parameter-space loads
      unsigned long long tl = 0ull;  // this row's occupied 64-column tiles
      // One 64-column group per iteration, kept as a loop (not unrolled) so the
      // epilogue's instructions stay in the instruction cache across groups.
#pragma unroll 1
      for (int gcol = 0; gcol < BN / 64; ++gcol) {
        const int nbase = g.n0 + gcol * 64;
        if (nbase >= p.N) break;  // uniform across the epilogue warps
        const int ncol0 = nbase + hf * 32;  // first column of this warp's block
        uint32_t stg = 0;
        if (!y_f32) {
          stg = stg_base + (uint32_t)((stg_count & 1) * kWarpStgBytes);
          if (lane == 0) bulk_wait_read<1>();  // the store that used this buffer has read it
          __syncwarp();
        }
        uint32_t raw[32];
        tmem_ld32_nowait(tbase + (uint32_t)(gcol * 64 + hf * 32), raw);
        tmem_wait_ld32(raw);
        if (KS > 1) {
          // the other units' partials of this row's 32 columns, in two halves:
          // every load of a half in flight before the first is used, added in
          // unit order
#pragma unroll
          for (int h = 0; h < 2; ++h) {
            float4 pv[kMaxSplit - 1][4];
#pragma unroll
            for (int k2i = 0; k2i < kMaxSplit - 1; ++k2i) {
              const int k2 = k2i < ks ? k2i : k2i + 1;
              if (k2 < KS) {
                const float4* src = reinterpret_cast<const float4*>(
                    ws_tile + ((int64_t)k2 * kBM + r) * BN + gcol * 64 + hf * 32 + h * 16);
#pragma unroll
                for (int i = 0; i < 4; ++i) pv[k2i][i] = __ldcg(src + i);
              }
            }
#pragma unroll
            for (int k2i = 0; k2i < kMaxSplit - 1; ++k2i) {
              const int k2 = k2i < ks ? k2i : k2i + 1;
              if (k2 < KS) {
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                  uint32_t* q4 = raw + h * 16 + 4 * i;
                  q4[0] = __float_as_uint(__uint_as_float(q4[0]) + pv[k2i][i].x);
                  q4[1] = __float_as_uint(__uint_as_float(q4[1]) + pv[k2i][i].y);
                  q4[2] = __float_as_uint(__uint_as_float(q4[2]) + pv[k2i][i].z);
                  q4[3] = __float_as_uint(__uint_as_float(q4[3]) + pv[k2i][i].w);
                }
              }
            }
          }
        }
        uint32_t rw = 0u;  // non-zero bits of this row in the warp's 32 columns
        const float* scg = scb + gcol * 64 + hf * 32;
        const float* shg = shb + gcol * 64 + hf * 32;
#pragma unroll
        for (int c16s = 0; c16s < 2; ++c16s) {
          const int nb = ncol0 + c16s * 16;
          const bool full = vec && (nb + 16 <= p.N);
          const float4* sc4 = reinterpret_cast<const float4*>(scg + c16s * 16);
          const float4* sh4 = reinterpret_cast<const float4*>(shg + c16s * 16);
          float o32[16];
          if (affine) {
#pragma unroll
            for (int q4 = 0; q4 < 4; ++q4) {
              const float4 sc = sc4[q4];
              const float4 sh = sh4[q4];
              o32[4 * q4 + 0] = fmaf(__uint_as_float(raw[c16s * 16 + 4 * q4 + 0]), sc.x, sh.x);
              o32[4 * q4 + 1] = fmaf(__uint_as_float(raw[c16s * 16 + 4 * q4 + 1]), sc.y, sh.y);
              o32[4 * q4 + 2] = fmaf(__uint_as_float(raw[c16s * 16 + 4 * q4 + 2]), sc.z, sh.z);
              o32[4 * q4 + 3] = fmaf(__uint_as_float(raw[c16s * 16 + 4 * q4 + 3]), sc.w, sh.w);
            }
          } else {
#pragma unroll
            for (int jj = 0; jj < 16; ++jj) o32[jj] = __uint_as_float(raw[c16s * 16 + jj]);
          }
          if (residual && mvalid) {
            const __nv_bfloat16* rp = residual + m * p.N + nb;
            if (full) {
              const uint4 r0 = *reinterpret_cast<const uint4*>(rp);
              const uint4 r1 = *reinterpret_cast<const uint4*>(rp + 8);
              const __nv_bfloat162* h0 = reinterpret_cast<const __nv_bfloat162*>(&r0);
              const __nv_bfloat162* h1 = reinterpret_cast<const __nv_bfloat162*>(&r1);
#pragma unroll
              for (int jj = 0; jj < 4; ++jj) {
                const float2 a0 = __bfloat1622float2(h0[jj]);
                const float2 a1 = __bfloat1622float2(h1[jj]);
                o32[2 * jj] += a0.x;
                o32[2 * jj + 1] += a0.y;
                o32[8 + 2 * jj] += a1.x;
                o32[8 + 2 * jj + 1] += a1.y;
              }
            } else {
              for (int jj = 0; jj < 16; ++jj)
                if (nb + jj < p.N) o32[jj] += __bfloat162float(rp[jj]);
            }
          }
          if (act == 1) {
#pragma unroll
            for (int jj = 0; jj < 16; ++jj) o32[jj] = fmaxf(o32[jj], 0.f);
          } else if (act == 2) {
#pragma unroll
            for (int jj = 0; jj < 16; ++jj) o32[jj] = fminf(fmaxf(o32[jj], 0.f), 6.f);
          } else if (act == 3) {
#pragma unroll
            for (int jj = 0; jj < 16; ++jj) o32[jj] = gelu_f(o32[jj]);
          }
          if (y_f32) {
            if (mvalid) {
              float* yp = reinterpret_cast<float*>(yout) + m * p.N + nb;
              if (full && (p.N % 4) == 0) {
#pragma unroll
                for (int jj = 0; jj < 16; jj += 4)
                  *reinterpret_cast<float4*>(yp + jj) = make_float4(o32[jj], o32[jj + 1], o32[jj + 2], o32[jj + 3]);
              } else {
                for (int jj = 0; jj < 16; ++jj)
                  if (nb + jj < p.N) yp[jj] = o32[jj];
              }
            }
          } else {
            uint32_t pk[8];
#pragma unroll
            for (int jj = 0; jj < 8; ++jj) {
              const __nv_bfloat162 h2 = __floats2bfloat162_rn(o32[2 * jj], o32[2 * jj + 1]);
              pk[jj] = *reinterpret_cast<const uint32_t*>(&h2);
            }
            if (emit) {
              uint32_t nzbits = 0u;
#pragma unroll
              for (int jj = 0; jj < 8; ++jj) {
                nzbits |= ((pk[jj] & 0x7FFFu) ? 1u : 0u) << (2 * jj);
                nzbits |= ((pk[jj] & 0x7FFF0000u) ? 1u : 0u) << (2 * jj + 1);
              }
              const int nvalid = p.N - nb;  // columns of this chunk inside the tensor
              if (!mvalid) nzbits = 0u;
              else if (nvalid < 16) nzbits &= nvalid > 0 ? ((1u << nvalid) - 1u) : 0u;
              rw |= nzbits << (c16s * 16);
            }
            // staging block: 32 rows x 64 bytes, 16-byte chunk k of row `lane` at
            // chunk k ^ ((lane >> 1) & 3) (the TMA 64-byte swizzle)
            const uint32_t row_addr = stg + (uint32_t)lane * 64u;
            const int k0 = c16s * 2;
            const int sx = (lane >> 1) & 3;
            sts_u4(row_addr + (uint32_t)((k0 ^ sx) << 4), make_uint4(pk[0], pk[1], pk[2], pk[3]));
            sts_u4(row_addr + (uint32_t)(((k0 + 1) ^ sx) << 4), make_uint4(pk[4], pk[5], pk[6], pk[7]));
          }
        }
        if (!y_f32) {
          fence_proxy_async_smem();
          __syncwarp();
          if (lane == 0) {
            tma_store_2d(&tmY, stg, ncol0, g.m0 + q * 32);
            bulk_commit();
          }
          ++stg_count;
        }
        if (emit) {
          // this block's share of the output occupancy
          if (rw) tl |= 1ull << ((nbase >> 6) & 63);
          const uint32_t bits = __reduce_or_sync(0xffffffffu, rw);
          if (lane == 0 && bits) atomicOr(&s_blk[gcol * 2 + hf], bits);  // the tile is the whole 128-row block
          // lane j: non-zeros of column 32 hf + j of this group in the warp's 32 rows
          s_cnt[q * BN + gcol * 64 + hf * 32 + lane] = __popc(warp_transpose32(rw));
        }
      }
      // accumulator b is free for the MMA of tile j + 2
      tc_fence_before();
      mbar_arrive(bar_acce + 8 * b);
      if (emit) {
        // both column halves of a row meet in shared memory; the half-0 thread of
        // the row then writes it once (a plain store when the tile spans every
        // column of the row's bitmap word, i.e. the word is this tile's alone)
        if (tl) atomicOr(&s_rowbm[r], tl);
        named_bar_sync(2, kEpiThreads);
        if (hf == 0) {
          const unsigned long long v = s_rowbm[r];
          s_rowbm[r] = 0ull;
          if (mvalid) {
            unsigned long long* dst = &o.row_bm[m * o.W64 + ((g.n0 >> 6) >> 6)];
            if (nt == 1) *dst = v;
            else if (v) atomicOr(dst, v);
          }
        }
        if (et < BN / 32) {
          const uint32_t v = s_blk[et];
          s_blk[et] = 0u;
          const int word = (g.n0 >> 5) + et;
          // rows m0.. m0+127 are one whole block and columns n0.. are this tile's
          if (word < o.C32) o.blk_mask[(g.m0 >> 7) * o.C32 + word] = v;
        }
        for (int c = et; c < BN; c += kEpiThreads) {
          const bool live = g.n0 + c < o.C;
          const uint32_t cnt =
              live ? s_cnt[c] + s_cnt[BN + c] + s_cnt[2 * BN + c] + s_cnt[3 * BN + c] : 0u;
          if (acc_smem) {
            if (live) s_acc[g.n0 + c] += cnt;  // one thread per column of this tile
          } else {
            if (cnt) atomicAdd(&o.col_nnz[g.n0 + c], cnt);
            uint32_t sum = cnt;
#pragma unroll
            for (int s = 16; s > 0; s >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, s);
            if (lane == 0 && sum) {
              atomicAdd(&o.tile_nnz[(g.n0 + c) >> 6], sum);
              atomicAdd(o.nnz, (unsigned long long)sum);
            }
          }
        }
      }
    }
    if (acc_smem) {
      // flush the CTA's column counts: per column, per 64-column tile, total
      named_bar_sync(2, kEpiThreads);
      const OccDev& o = P.out_occ;
      unsigned long long total = 0ull;
      for (int c0 = 0; c0 < p.N; c0 += kEpiThreads) {
        const int c = c0 + et;
        const uint32_t cnt = c < p.N ? s_acc[c] : 0u;
        if (cnt) atomicAdd(&o.col_nnz[c], cnt);
        uint32_t sum = cnt;
#pragma unroll
        for (int s = 16; s > 0; s >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, s);
        total += sum;
        if (lane == 0 && sum) atomicAdd(&o.tile_nnz[c >> 6], sum);
      }
      if (lane == 0 && total) atomicAdd(o.nnz, total);
    }
    if (lane == 0) bulk_wait_all();
  }

  __syncwarp();  // lanes that finished early wait for their warp's working lane
  tc_fence_before();
  __syncthreads();
  if (*s_abort) {
    // a bounded wait ran out: before shared and tensor memory are released,
    // the copies into the last stage of every ring slot have landed and the
    // MMAs issued so far are done (each wait bounded again)
    if (threadIdx.x == 0) {
      const int issued = *s_issued;
      if (resident_b) mbar_drain(bar_resb, 0u, wlim);
      for (int k = 0; k < S && k < issued; ++k) {
        const int i = issued - 1 - k;
        mbar_drain(bar_full + 8 * (i % S), (uint32_t)((i / S) & 1), wlim);
      }
    }
    if (warp == kMmaWarp && elect_one()) {
      tc_commit(bar_drain);
      mbar_drain(bar_drain, 0u, wlim);
    }
    __syncthreads();
  }
  if (warp == kMmaWarp) {
    tc_fence_after();
    tmem_dealloc(tmem, kTmemCols);
  }
}

// ---------------------------------------------------------------------------
// Host side
// ---------------------------------------------------------------------------
}  // namespace

PFN_cuTensorMapEncodeTiled_v12000 tmap_encoder() {
  static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
  static std::once_flag once;
  std::call_once(once, [] {
    void* ptr = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &ptr, 12000, cudaEnableDefault,
                                         &q) == cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(ptr);
  });
  return fn;
}

static CUtensorMapSwizzle swz_of(int inner_bytes) {
  return inner_bytes == 128 ? CU_TENSOR_MAP_SWIZZLE_128B : CU_TENSOR_MAP_SWIZZLE_64B;
}

// 2-D bf16 tensor [rows, cols] (cols contiguous), box {box_cols, box_rows}.
bool make_tmap_2d(CUtensorMap* m, const void* base, uint64_t rows, uint64_t cols, uint32_t box_cols,
                  uint32_t box_rows) {
  auto enc = tmap_encoder();
  if (!enc) return false;
  cuuint64_t dims[2] = {cols, rows};
  cuuint64_t strides[1] = {cols * 2};
  cuuint32_t box[2] = {box_cols, box_rows};
  cuuint32_t estr[2] = {1, 1};
  CUresult r = enc(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(base), dims, strides,
                   box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE, swz_of((int)box_cols * 2),
                   CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS;
}

// 4-D NHWC bf16 tensor [n, h, w, c], box {box_c, bw, bh, bn} traversed with
// element strides {1, stride, stride, 1}.
bool make_tmap_nhwc(CUtensorMap* m, const void* base, int n, int h, int w, int c, int box_c, int bw,
                    int bh, int bn, int stride) {
  auto enc = tmap_encoder();
  if (!enc) return false;
  cuuint64_t dims[4] = {(cuuint64_t)c, (cuuint64_t)w, (cuuint64_t)h, (cuuint64_t)n};
  cuuint64_t strides[3] = {(cuuint64_t)c * 2, (cuuint64_t)w * c * 2, (cuuint64_t)h * w * c * 2};
  cuuint32_t box[4] = {(cuuint32_t)box_c, (cuuint32_t)(bw * stride), (cuuint32_t)(bh * stride),
                       (cuuint32_t)bn};
  cuuint32_t estr[4] = {1, (cuuint32_t)stride, (cuuint32_t)stride, 1};
  CUresult r = enc(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, const_cast<void*>(base), dims, strides,
                   box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE, swz_of(box_c * 2),
                   CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS;
}

namespace {

template <int BN, int BK, int LEAN, bool STEM = false>
cudaError_t launch_cfg(const IgemmArgs& a, const CUtensorMap& tA, const CUtensorMap& tB,
                       const CUtensorMap& tY, const CUtensorMap& tA32, const CUtensorMap& tB32,
                       int64_t tiles, cudaStream_t s) {
  cudaError_t e0 =
      smem_optin(reinterpret_cast<const void*>(igemm_kernel<BN, BK, LEAN, STEM>), (size_t)Cfg<BN, BK, STEM>::kSmem);
  if (e0 != cudaSuccess) return e0;
  const int64_t units = tiles * (a.ksplit > 1 ? a.ksplit : 1);
  const int64_t grid = units < device_sm_count() ? units : device_sm_count();
  cudaError_t e = launch_kernel(igemm_kernel<BN, BK, LEAN, STEM>, dim3((unsigned)grid), dim3(Warps<LEAN, STEM>::kThreads),
                                (size_t)Cfg<BN, BK, STEM>::kSmem, s, tA, tB, tY, tA32, tB32, a);
  if (e != cudaSuccess) return e;
  return cudaGetLastError();
}

template <int LEAN>
cudaError_t launch_bn(const IgemmArgs& a, int bn, int bk, const CUtensorMap& tA, const CUtensorMap& tB,
                      const CUtensorMap& tY, const CUtensorMap& tA32, const CUtensorMap& tB32, int64_t tiles,
                      cudaStream_t s) {
  if (bk == 64) {
    switch (bn) {
      case 64: return launch_cfg<64, 64, LEAN>(a, tA, tB, tY, tA32, tB32, tiles, s);
      case 96:
        if constexpr (LEAN) return launch_cfg<96, 64, LEAN>(a, tA, tB, tY, tA32, tB32, tiles, s);
        return cudaErrorInvalidValue;  // (choose_tiles: lean kernels only)
      case 160:
        if constexpr (LEAN) return launch_cfg<160, 64, LEAN>(a, tA, tB, tY, tA32, tB32, tiles, s);
        return cudaErrorInvalidValue;
      case 128: return launch_cfg<128, 64, LEAN>(a, tA, tB, tY, tA32, tB32, tiles, s);
      case 192: return launch_cfg<192, 64, LEAN>(a, tA, tB, tY, tA32, tB32, tiles, s);
      default: return launch_cfg<256, 64, LEAN>(a, tA, tB, tY, tA32, tB32, tiles, s);
    }
  }
  switch (bn) {
    case 64: return launch_cfg<64, 32, LEAN>(a, tA, tB, tY, tA32, tB32, tiles, s);
    case 128: return launch_cfg<128, 32, LEAN>(a, tA, tB, tY, tA32, tB32, tiles, s);
    case 192: return launch_cfg<192, 32, LEAN>(a, tA, tB, tY, tA32, tB32, tiles, s);
    default: return launch_cfg<256, 32, LEAN>(a, tA, tB, tY, tA32, tB32, tiles, s);
  }
}

}  // namespace


void choose_spatial_tile(IgemmArgs& a) {
  int64_t best = -1;
  for (int bw = 1; bw <= 128; bw *= 2) {
    if (bw * a.stride > 256) break;
    for (int bh = 1; bw * bh <= 128; bh *= 2) {
      if (bh * a.stride > 256) break;
      const int bn = 128 / (bw * bh);
      const int64_t tw = (a.Wo + bw - 1) / bw, th = (a.Ho + bh - 1) / bh,
                    tn = (a.Nimg + bn - 1) / bn;
      const int64_t cost = tw * bw * th * bh * tn * bn;
      // fewest padded pixels; then the widest (most contiguous) box
      if (best < 0 || cost < best || (cost == best && bw > a.bw)) {
        best = cost;
        a.bw = bw;
        a.bh = bh;
        a.bn = bn;
        a.tw = (int)tw;
        a.th = (int)th;
      }
    }
  }
}

// N tile and K split.  The main loop is bound by shared-memory traffic: a
// K block of a 128 x BN tile is written by TMA and read back by the MMAs,
// (128 + BN) rows each way, so a tile costs about (128 + BN) per K block and
// the tiles take ceil(tiles / SMs) rounds over the SMs.  Of 96, 128, 160, 192
// and 256 wide tiles the cheapest total wins, ties going to 128 and then to the
// narrower (a shorter epilogue); 64 wide ones when 128 wide tiles would fill under
// half of the SMs.  On GB300, GEMMs with M 1024..8192, K 768..3072 and N
// 768..3072 follow this ordering.  96 and 160: lean kernels with 64-wide K blocks;
// with weights in L2 they gain little (1576 rows x 3072 columns 11.9 -> 11.5 us),
// with weights from memory the additional CTAs have
// more loads in flight (ViT-B/16 at batch 8, 1576 rows: 1175 -> 1139 us).  K blocks are 64 wide (128-byte swizzle) wherever the
// channel layout allows: 32 wide ones were slower at every tile width.
// 64-wide tiles that number at most the SMs go to the one-tile-per-cluster
// kernel (k_onetile.cu), which shares a tile's K range through distributed
// shared memory.  The gather mode, which that kernel does not have, splits K
// here while the tiles leave SMs idle, at most 4 ways and with at least 8 K
// blocks per unit (the tile's last unit reads the other partials alone).
static int k_block(const IgemmArgs& a) { return (a.conv == 2 ? (a.Cp % 64 == 0) : (a.Ktot > 32)) ? 64 : 32; }

void choose_tiles(const IgemmArgs& a, int64_t mtiles, bool lean, int* bn_out, int* ks_out) {
  const int sms = device_sm_count();
  int bn = a.N > 64 ? 128 : 64;
  int64_t tiles = mtiles * ((a.N + bn - 1) / bn);
  if (bn == 128 && tiles < sms / 2) {
    bn = 64;
    tiles = mtiles * ((a.N + bn - 1) / bn);
  } else if (bn == 128) {
    int64_t best = ((tiles + sms - 1) / sms) * (128 + 128);
    for (const int cand : {96, 160, 192, 256}) {
      if (cand >= a.N + 64) break;
      if (cand != 256 && a.N > 4096) continue;  // a tile's columns lie in one word of the row bitmap
      if (cand % 64 && !(lean && k_block(a) == 64)) continue;
      const int64_t t = mtiles * ((a.N + cand - 1) / cand);
      const int64_t cost = ((t + sms - 1) / sms) * (128 + cand);
      if (cost < best) {
        best = cost;
        bn = cand;
        tiles = t;
      }
    }
  }
  const int bk = k_block(a);
  const int kblocks = (a.Ktot + bk - 1) / bk;
  int ks = 1;
  if (a.conv == 1 && a.ws && a.ws_cnt && tiles < sms && tiles <= a.ws_cnt_len) {
    ks = (int)(sms / tiles);
    if (ks > kMaxSplit) ks = kMaxSplit;
    while (ks > 1 && (kblocks < 8 * ks || (size_t)tiles * ks * kBM * bn * 4 > a.ws_bytes)) --ks;
  }
  *bn_out = bn;
  *ks_out = ks;
}

// n / d = umulhi(n, mul) >> shift for 0 <= n < 2^31 (Granlund and Montgomery,
// "Division by invariant integers using multiplication", 1994: with 2^l >= d,
// mul = ceil(2^(31 + l) / d) < 2^32 and the product's excess stays below 2^(31+l)/d).
static void div_magic(uint32_t d /* >= 2 */, uint32_t* mul, uint32_t* shift) {
  uint32_t l = 0;
  while ((1u << l) < d) ++l;
  const uint64_t num = (uint64_t)1 << (31 + l);
  *mul = (uint32_t)((num + d - 1) / d);
  *shift = l - 1;
}

bool stem_plan(const __nv_bfloat16* x, int64_t n, int H, int W, int C, int N, int kh, int kw, int stride, int pad,
               StemGeo* g) {
  StemGeo q;
  q.x = x;
  q.H = H;
  q.W = W;
  q.C = C;
  q.kh = kh;
  q.kw = kw;
  q.stride = stride;
  q.pad = pad;
  q.Ho = (H + 2 * pad - kh) / stride + 1;
  q.Wo = (W + 2 * pad - kw) / stride + 1;
  if (C >= 8 || kh * kw <= 1 || N > 64 || N % 8 || n <= 0) return false;
  // a window of a kernel row fits 24 K columns, the whole window three K blocks
  if (kw * C > 24 || pad >= kw || pad >= kh) return false;
  q.seg = (kw * C + 7) / 8 * 8;
  if (kh * q.seg > 192) return false;
  // a tile's 128 pixels lie in at most two images
  if ((int64_t)q.Ho * q.Wo < kBM || (int64_t)n * q.Ho * q.Wo > ((int64_t)1 << 31) - 1 - kBM) return false;
  const int span = 1 + (kBM - 1 + q.Wo - 1) / q.Wo;
  const int one = kh + (span - 1) * stride, two = 2 * kh + (span - 2) * stride;
  q.rows = one > two ? one : two;
  q.lead = (pad * C + 1 + 7) / 8 * 8;
  const int need = q.lead + 7 + (W * C > (q.Wo - 1) * stride * C ? W * C : (q.Wo - 1) * stride * C) + q.seg + 10;
  q.pitch = (need + 7) / 8 * 8;
  if (q.rows > kMaxStemRows || (int64_t)q.rows * q.pitch * 2 > kStemRowBytes || (int64_t)W * stride * C >= (1 << 23)) return false;
  if (q.Wo < 2 || q.Ho < 2) return false;  // (a divisor of 1 has no 32-bit multiplier)
  div_magic((uint32_t)q.Wo, &q.wo_mul, &q.wo_shift);
  div_magic((uint32_t)q.Ho, &q.ho_mul, &q.ho_shift);
  q.ragged = (reinterpret_cast<uintptr_t>(x) & 15u) != 0 || (W * C) % 8 != 0;
  *g = q;
  return true;
}

cudaError_t launch_igemm(const IgemmArgs& a_in, cudaStream_t s) {
  IgemmArgs a = a_in;
  if (a.M <= 0 || a.N <= 0) return cudaSuccess;
  if (a.stem.x) {
    CUtensorMap tB, tY;
    if (!make_tmap_2d(&tB, a.w, (uint64_t)a.N, (uint64_t)a.Ktot, 64, 64) ||
        !make_tmap_2d(&tY, a.y, (uint64_t)a.M, (uint64_t)a.N, 32, 32))
      return cudaErrorInvalidValue;
    const int64_t tiles = ((int64_t)a.M + kBM - 1) / kBM;
    return a.ep.residual ? launch_cfg<64, 64, 2, true>(a, tB, tB, tY, tB, tB, tiles, s)
                         : launch_cfg<64, 64, 1, true>(a, tB, tB, tY, tB, tB, tiles, s);
  }
  if (a.conv == 2 && (a.Cp % 32 != 0 || a.bw * a.bh * a.bn != 128)) return cudaErrorInvalidValue;
  if (a.conv == 2 && (reinterpret_cast<uintptr_t>(a.ep.residual) & 15u) != 0) return cudaErrorInvalidValue;  // (lean kernels only)
  const int64_t mtiles =
      a.conv == 2 ? (int64_t)((a.Nimg + a.bn - 1) / a.bn) * a.th * a.tw : (a.M + kBM - 1) / kBM;
  int bn = 64, ks = 1;
  const bool lean = a.conv != 1 && !a.y_f32 && !a.dense_only &&
                    (a.ep.residual == nullptr ||
                     (a.N % 8 == 0 && (reinterpret_cast<uintptr_t>(a.ep.residual) & 15u) == 0));
  choose_tiles(a, mtiles, lean, &bn, &ks);
  a.ksplit = ks;
  const int bk = k_block(a);
  if (bn == 64) {
    const int split = onetile_split(a, mtiles, bk, lean);
    if (split > 0) {
      a.ksplit = split;
      return launch_onetile(a, mtiles, bk, s);
    }
  }
  CUtensorMap tA, tB, tY;
  memset(&tA, 0, sizeof(tA));
  memset(&tY, 0, sizeof(tY));
  if (a.conv == 0) {
    if (!make_tmap_2d(&tA, a.x, (uint64_t)a.M, (uint64_t)a.Ktot, (uint32_t)bk, kBM))
      return cudaErrorInvalidValue;
  } else if (a.conv == 2) {
    if (!make_tmap_nhwc(&tA, a.x, a.Nimg, a.H, a.W, a.Cp, bk, a.bw, a.bh, a.bn, a.stride))
      return cudaErrorInvalidValue;
  }
  if (!make_tmap_2d(&tB, a.w, (uint64_t)a.N, (uint64_t)a.Ktot, (uint32_t)bk, (uint32_t)bn))
    return cudaErrorInvalidValue;
  if (!a.y_f32) {
    // one epilogue warp's block: 32 columns x 32 tile rows (for spatial tiles
    // the sub-box {bw', bh', bn'} of 32 pixels that the rows form)
    const int sbw = a.bw < 32 ? a.bw : 32;
    const int sbh = a.bh < 32 / sbw ? a.bh : 32 / sbw;
    const int sbn = 32 / (sbw * sbh);
    bool okY = a.conv == 2
                   ? make_tmap_nhwc(&tY, a.y, a.Nimg, a.Ho, a.Wo, a.N, 32, sbw, sbh, sbn, 1)
                   : make_tmap_2d(&tY, a.y, (uint64_t)a.M, (uint64_t)a.N, 32, 32);
    if (!okY) return cudaErrorInvalidValue;
  }
  if (a.conv == 1) tA = tB;  // unused by the gather producers
  // 32-column boxes (64-byte swizzle) of the compacted zero-skip GEMM
  CUtensorMap tA32 = tB, tB32 = tB;
  if (a.conv == 0 && bk == 64) {
    if (!make_tmap_2d(&tA32, a.x, (uint64_t)a.M, (uint64_t)a.Ktot, 32, kBM) ||
        !make_tmap_2d(&tB32, a.w, (uint64_t)a.N, (uint64_t)a.Ktot, 32, (uint32_t)bn))
      return cudaErrorInvalidValue;
  }
  const int64_t tiles = mtiles * ((a.N + bn - 1) / bn);
  if (!lean) return launch_bn<0>(a, bn, bk, tA, tB, tY, tA32, tB32, tiles, s);
  return a.ep.residual ? launch_bn<2>(a, bn, bk, tA, tB, tY, tA32, tB32, tiles, s)
                       : launch_bn<1>(a, bn, bk, tA, tB, tY, tA32, tB32, tiles, s);
}

}  // namespace sparoa
