// Dense and zero-skipping implicit GEMM for problems with fewer 128 x 64 output
// tiles than SMs (batch-1 networks, late CNN stages, short token counts):
// one tile per thread-block cluster, its K range shared by the cluster's CTAs.
//
// Such a launch is a chain of latencies, not bound by any rate: a handful of K
// blocks per CTA, then the sum over the K shares, then the epilogue.  Against
// the persistent kernel with its split K through global memory: ResNet-18 at
// batch 1 311 -> 177 us, a strided basic block at batch 8 (28x28x128 -> 14x14x256,
// three convolutions) 47 -> 33 us when it came, 173 and 28 us now; one call (with its occupancy clear) 8.1 us on [1,14,14,256]
// 3x3 and 9.2 us on [1,7,7,512] 3x3, of which (clock64) 1.2 us to the first
// operands, 0.5-1.5 us of MMAs, 0.4 us to read the accumulator, 0.6 us at the
// cluster barrier, 1.2 us for the sum and the stores, 0.7 us of occupancy.  So
//   - the K range of a tile is cut over up to 8 CTAs of one cluster, and the
//     fp32 partial tiles meet in distributed shared memory: no partials in
//     global memory, no arrival tickets, no CTA left with the whole epilogue;
//   - every CTA of the cluster adds up and finishes every KS-th row of the tile
//     (shares in rank order, so results do not depend on timing), a thread
//     4 columns of one row, so output rows leave as whole 128-byte lines and
//     the occupancy bits come from ballots;
//   - the stages of the ring are issued by one warp each, all at once, and a
//     spatial tile's box covers only the images that exist;
//   - one short code path: a CTA runs every instruction about once, so the
//     instruction cache misses of a long epilogue are paid in full.
#include <cuda.h>

#include <cstring>
#include <mutex>

#include "igemm_geo.cuh"
#include "sparoa_kernels.h"

namespace sparoa {

namespace {

constexpr int kBN = 64;
constexpr int kWarps = 8;                     // producers, then epilogue
constexpr int kWorkers = 32 * kWarps;
constexpr int kThreads = kWorkers + 32;       // + the MMA warp
constexpr int kStages = kWarps;               // stage s is filled by warp s
constexpr int kMaxItems = 2048;               // K blocks of a CTA's share (more: another kernel)
constexpr int kMaxTapsHere = 64;
constexpr int kPitch = kBN + 4;               // floats per row of the partial tile
constexpr uint32_t kTmemCols = 64;

template <int BK>
struct Lay {
  static constexpr int kA = kBM * BK * 2;
  static constexpr int kB = kBN * BK * 2;
  static constexpr int kStage = kA + kB;
  static constexpr int kRing = kStages * kStage;
  static constexpr int kPart = kBM * kPitch * 4;  // overlays the ring once the MMAs are done
  static constexpr int kBar = kRing > kPart ? kRing : kPart;
  static constexpr int kNumBars = 2 * kStages + 2;  // full, empty, accumulator, drain
  static constexpr int kFlag = kBar + kNumBars * 8;  // abort, tmem, items, issued[kStages]
  static constexpr int kBits = kFlag + (3 + kStages) * 4 + 4;
  static constexpr int kTap = (kBits + 2 * kMaxItems / 8 + 7) & ~7;
  static constexpr int kItems = kTap + kMaxTapsHere * 8;
  static constexpr int kCnt = kItems + kMaxItems * 2;
  static constexpr int kWord = kCnt + kBN * 4;  // [rows of the share][2] non-zero bits
  static constexpr int kBytes = kWord + kBM * 2 * 4;
  static constexpr int kSmem = kBytes + 1024;
  static_assert(kSmem <= 227 * 1024, "shared memory");
};

__device__ __forceinline__ float4 ld_cluster_f4(uint32_t addr) {
  float4 v;
  asm volatile("ld.shared::cluster.v4.f32 {%0, %1, %2, %3}, [%4];"
               : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w)
               : "r"(addr)
               : "memory");
  return v;
}

template <int BK, int KS>
__global__ void __launch_bounds__(kThreads, 1)
    onetile_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB,
                   const IgemmArgs P, const int a_rows) {
  using L = Lay<BK>;
  // rows of the tile this CTA finishes: rank, rank + KS, ... (interleaved, so
  // that a tile's missing rows are shared evenly)
  constexpr int kRows = kBM / KS;
  constexpr int kIters = kRows * 16 / kWorkers;  // a thread: 4 columns of kIters rows, 16 rows apart
  const Geo p = make_geo(P);
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  const uint32_t sbase = smem_u32(smem);
  const uint32_t bar_full = sbase + L::kBar;
  const uint32_t bar_empty = bar_full + 8 * kStages;
  const uint32_t bar_acc = bar_empty + 8 * kStages;
  const uint32_t bar_drain = bar_acc + 8;
  int* flags = reinterpret_cast<int*>(smem + L::kFlag);
  volatile int* s_abort = flags;
  uint32_t* s_tmem = reinterpret_cast<uint32_t*>(flags + 1);
  volatile int* s_nitems = flags + 2;
  volatile int* s_issued = flags + 3;  // [kStages] fills of stage s so far
  // occupied K blocks of the share: their first and their last 32 columns
  uint32_t* s_lo = reinterpret_cast<uint32_t*>(smem + L::kBits);
  uint32_t* s_hi = s_lo + kMaxItems / 32;
  unsigned long long* s_tap = reinterpret_cast<unsigned long long*>(smem + L::kTap);
  uint16_t* s_items = reinterpret_cast<uint16_t*>(smem + L::kItems);
  uint32_t* s_cnt = reinterpret_cast<uint32_t*>(smem + L::kCnt);
  uint32_t* s_word = reinterpret_cast<uint32_t*>(smem + L::kWord);
  const int warp = threadIdx.x >> 5;
  const int lane = threadIdx.x & 31;
  const long long wlim = P.wait_limit > 0 ? P.wait_limit : kWaitLimitCycles;
  uint32_t* const err = P.err;
  const int tile = (int)blockIdx.x / KS;
  const int rank = (int)blockIdx.x % KS;  // rank in the cluster (KS consecutive CTAs)

  if (P.dense_only) {
    // launched next to the small-FC kernel, which handles the zero-skip path
    pdl_wait();
    if (decide_path(P.disp) == 2) {
      pdl_trigger();
      return;
    }
  }
  // ---- on-chip set-up and everything that follows from the parameters alone
  if (threadIdx.x < kStages) {
    mbar_init(bar_full + 8 * threadIdx.x, 1u);
    mbar_init(bar_empty + 8 * threadIdx.x, 1u);
    s_issued[threadIdx.x] = 0;
    if (threadIdx.x == 0) {
      mbar_init(bar_acc, 1u);
      mbar_init(bar_drain, 1u);
      *s_abort = 0;
    }
    fence_mbar_init();
  }
  if (threadIdx.x == kWorkers) {
    prefetch_tmap(&tmA);
    prefetch_tmap(&tmB);
  }
  if (warp == kWarps) tmem_alloc(smem_u32(s_tmem), kTmemCols);
  if (threadIdx.x == kWorkers + 1) s_lo[0] = 0u;
  if (threadIdx.x < kBN) s_cnt[threadIdx.x] = 0u;
  if (threadIdx.x >= 64 && threadIdx.x < 64 + kMaxTapsHere) s_tap[threadIdx.x - 64] = 0ull;
  const int kblocks = (p.Ktot + BK - 1) / BK;
  const int kb0 = (int)((int64_t)rank * kblocks / KS);
  const int span = (int)((int64_t)(rank + 1) * kblocks / KS) - kb0;  // K blocks of this CTA's share
  const int lap = span < kStages ? span : kStages;                   // ... of which one ring full at most
  const int nt = (p.N + kBN - 1) / kBN;
  const TileGeo g = tile_geo(p, tile, nt, kBN);
  const int cbpt = p.conv == 2 ? p.Cp / BK : 1;  // channel blocks per tap
  const int y0 = g.th0 * p.stride - p.pad, x0 = g.tw0 * p.stride - p.pad;
  const uint32_t fb = bar_full + 8 * warp;
  const uint32_t sa = sbase + warp * L::kStage;
  // K block kb into stage `warp`: operand B (the weights), operand A
  auto load_b = [&](int kb) { tma_load_2d(sa + L::kA, &tmB, fb, kb * BK, g.n0); };
  int ac, ax, ay;  // operand A's next box: channel, column, row (GEMM: channel, row)
  auto seek_a = [&](int kb) {
    if (p.conv == 0) {
      ac = kb * BK;
      ax = 0;
      ay = g.m0;
    } else {
      const int tp = kb / cbpt;
      ac = (kb - tp * cbpt) * BK;
      ay = tp / p.kw;
      ax = x0 + tp - ay * p.kw;
      ay += y0;
    }
  };
  auto load_a = [&]() {
    if (p.conv == 0) tma_load_2d(sa, &tmA, fb, ac, ay);
    else tma_load_4d(sa, &tmA, fb, ac, ax, ay, g.tn0);
  };
  seek_a(kb0 + warp);
  const uint32_t stage_bytes = (uint32_t)((a_rows + kBN) * BK * 2);
  const bool has_bits = p.conv == 0 ? P.in_blk != nullptr
                                    : (P.in_rowbm != nullptr && P.in_W64 == 1 && p.kh * p.kw <= kMaxTapsHere);
  const bool masks = has_bits && P.disp.force != 1 && warp < kWarps;
  const uint32_t* const words = p.conv == 0 && has_bits ? P.in_blk + (int64_t)(g.m0 >> 7) * P.in_C32 : nullptr;
  // a convolution's share: this thread's taps from tap0 on in steps of 2, up to t1
  int tap0 = 0, t1 = -1;
  const uint64_t* px = nullptr;  // row words at the origin of this thread's pixel's window
  int iy = 0, ix = 0;
  uint32_t inv_kw = 0u;          // tap / kw = tap * inv_kw >> 16 (taps < 64)
  if (masks && p.conv == 2) {
    tap0 = kb0 / cbpt + ((int)threadIdx.x >> 7);
    t1 = (kb0 + span - 1) / cbpt;
    inv_kw = 65536u / (uint32_t)p.kw + 1u;
    bool pv;
    int pn, oy, ox;
    tile_row(p, g, threadIdx.x & 127, pv, pn, oy, ox);
    iy = oy * p.stride - p.pad;
    ix = ox * p.stride - p.pad;
    if (pv) px = reinterpret_cast<const uint64_t*>(P.in_rowbm) + ((int64_t)pn * p.H + iy) * p.W + ix;
  }
  auto load_tap = [&](int tap) -> unsigned long long {
    const int tr = (int)((uint32_t)tap * inv_kw >> 16), tc = tap - tr * p.kw;
    if (px && tap <= t1 && (unsigned)(iy + tr) < (unsigned)p.H && (unsigned)(ix + tc) < (unsigned)p.W)
      return px[tr * p.W + tc];
    return 0ull;
  };
  // output rows and column affine of this thread
  const int c4 = threadIdx.x & 15;
  const int col = g.n0 + 4 * c4;
  const bool cvalid = warp < kWarps && col < p.N;  // N % 8 == 0: all 4 columns or none
  int mrow[kIters];                                // output row, -1: none
#pragma unroll
  for (int i = 0; i < kIters; ++i) {
    bool v;
    int img, oh, ow;
    const int64_t m = tile_row(p, g, (i * 16 + ((int)threadIdx.x >> 4 & 15)) * KS + rank, v, img, oh, ow);
    mrow[i] = v && cvalid ? (int)m : -1;
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *s_tmem;
  if (P.early_w && warp < lap && lane == 0) {  // the weights are complete: their first ring full is requested now
    mbar_arrive_expect_tx(fb, stage_bytes);
    load_b(kb0 + warp);
  }
  pdl_wait();
  pdl_trigger();
  if (warp < lap && lane == 0) {
    if (!P.early_w) {
      mbar_arrive_expect_tx(fb, stage_bytes);
      load_b(kb0 + warp);
    }
    load_a();
    s_issued[warp] = 1;
  }
  // ---- zero-skip path: the occupied K blocks.  The first ring full is loaded
  // whatever it holds (the masks arrive no sooner than the blocks), of the rest
  // of the share only occupied blocks; empty blocks, and the empty half of a
  // GEMM's block (32 columns), are not multiplied.  The masks' first loads are
  // on their way before the rule is known.  (Short, rolled code: a CTA runs it
  // once, and every eight instructions cost an instruction cache miss.)
  unsigned long long w = 0ull;
  if (masks && p.conv == 2) w = load_tap(tap0);
  uint32_t glo = 0u, ghi = 0u;
  auto load_words = [&](int i0) {  // the mask words of K block i0 + lane of the share
    const int b = kb0 + i0 + lane;
    glo = ghi = 0u;
    if (i0 + lane < span) {
      glo = words[b * (BK / 32)];
      if (BK == 64 && 2 * b + 1 < P.in_C32) ghi = words[2 * b + 1];
    }
  };
  if (masks && p.conv == 0) load_words(warp * 32);
  const int path = decide_path(P.disp);
  record_path(P.disp, path);
  const bool listed = path == 2 && has_bits;
  if (listed && warp < kWarps) {
    // nothing but occupied blocks is added to the accumulator
    tmem_st32_zero(tmem + ((uint32_t)((warp & 3) * 32) << 16) + (uint32_t)((warp >> 2) * 32));
    if (p.conv == 2) {
      // per tap of the share: the occupied 64-channel tiles over the tile's pixels
      const bool direct = BK == 64 && span <= 32;  // a tile is a K block: its bit at once
#pragma unroll 1
      for (int tp = tap0; tp <= t1; tp += 2) {
        const unsigned long long ahead = load_tap(tp + 2);
        const uint32_t lo = __reduce_or_sync(0xffffffffu, (uint32_t)w);
        const uint32_t hi = __reduce_or_sync(0xffffffffu, (uint32_t)(w >> 32));
        const unsigned long long ww = ((unsigned long long)hi << 32) | lo;
        const int sh = tp * cbpt - kb0;
        if (lane == 0 && ww) {
          if (direct) atomicOr(&s_lo[0], (uint32_t)(sh >= 0 ? ww << sh : ww >> -sh) & (0xFFFFFFFFu >> (32 - span)));
          else atomicOr(&s_tap[tp], ww);
        }
        w = ahead;
      }
      if (!direct) {
        named_bar_sync(1, kWorkers);
        for (int i0 = warp * 32; i0 < span; i0 += kWorkers) {
          const int b = kb0 + i0 + lane, tp = b / cbpt;
          const uint32_t bits = __ballot_sync(
              0xffffffffu, i0 + lane < span && ((s_tap[tp] >> (((b - tp * cbpt) * BK) >> 6)) & 1ull) != 0ull);
          if (lane == 0) s_lo[i0 >> 5] = bits;
        }
      }
    } else {
      for (int i0 = warp * 32; i0 < span; i0 += kWorkers) {
        if (i0 >= kWorkers) load_words(i0);
        const uint32_t lo = __ballot_sync(0xffffffffu, glo != 0u), hi = __ballot_sync(0xffffffffu, ghi != 0u);
        if (lane == 0) {
          s_lo[i0 >> 5] = lo;
          s_hi[i0 >> 5] = hi;
        }
      }
    }
    if (span > 32) {  // (up to 32 blocks, the one word is the list)
      named_bar_sync(1, kWorkers);
      if (warp == 0) {
        int n = 0;
        for (int w32 = 0; w32 * 32 < span; ++w32) {
          uint32_t bits = p.conv == 2 ? s_lo[w32] : s_lo[w32] | s_hi[w32];
          if (w32 == 0) bits &= ~((1u << kStages) - 1u);
          if ((bits >> lane) & 1u) s_items[n + __popc(bits & ((1u << lane) - 1u))] = (uint16_t)(w32 * 32 + lane);
          n += __popc(bits);
        }
        if (lane == 0) *s_nitems = n;
      }
    }
    tmem_wait_st();
    tc_fence_before();
  }
  // after the list's barrier: the occupied blocks behind the first ring full
  auto listed_rest = [&]() -> int {
    if (span > 32) return *s_nitems;
    return __popc((p.conv == 2 ? s_lo[0] : s_lo[0] | s_hi[0]) & ~((1u << kStages) - 1u));
  };
  auto listed_block = [&](int i) -> int {
    if (span > 32) return (int)s_items[i];
    uint32_t bits = (p.conv == 2 ? s_lo[0] : s_lo[0] | s_hi[0]) & ~((1u << kStages) - 1u);
    for (; i > 0; --i) bits &= bits - 1u;
    return __ffs(bits) - 1;
  };
  if (warp == kWarps) {
    // ------------------------------------------------------------------ MMA issue
    constexpr uint32_t idesc = idesc_bf16_f32(kBM, kBN);
    const bool el = elect_one();
    const uint64_t ad = smem_desc_kmajor<BK>(sbase), bd = smem_desc_kmajor<BK>(sbase + L::kA);
    bool ok = true;
    uint32_t ph = 0u;
    // (the dense path's stages s = i % 8 are unrolled: the descriptors are
    // constants from the base)
    if (!listed) {
      for (int i0 = 0; ok && i0 < span; i0 += kStages) {
#pragma unroll
        for (int s = 0; s < kStages; ++s) {
          if (ok && i0 + s < span) {
            ok = mbar_wait_warp(bar_full + 8 * s, ph, err, s_abort, kErrTimeoutFull, wlim);
            if (ok) {
              tc_fence_after();
              const uint64_t a = ad + (uint64_t)(s * (L::kStage / 16)), b = bd + (uint64_t)(s * (L::kStage / 16));
              if (el) {
                if (s == 0 && i0 == 0) tc_mma_bf16(tmem, a, b, idesc, 0u);
                else tc_mma_bf16(tmem, a, b, idesc, 1u);
#pragma unroll
                for (int k = 1; k < BK / 16; ++k) tc_mma_bf16(tmem, a + (uint64_t)(2 * k), b + (uint64_t)(2 * k), idesc, 1u);
                tc_commit(bar_empty + 8 * s);
              }
            }
            __syncwarp();
          }
        }
        ph ^= 1u;
      }
    } else {
      // the first ring full, whatever the masks say in each stage (rolled: a
      // block's code once), into an accumulator of zeros
      named_bar_sync(2, kThreads);  // the list is complete
      tc_fence_after();
      const uint32_t wlo = s_lo[0], whi = p.conv == 2 ? wlo : s_hi[0];
      const int total = lap + listed_rest();
      uint64_t a = ad, b = bd;
#pragma unroll 1
      for (int s = 0; ok && s < lap; ++s) {
        ok = mbar_wait_warp(bar_full + 8 * s, 0u, err, s_abort, kErrTimeoutFull, wlim);
        if (ok) {
          tc_fence_after();
          if (el) {
            if ((wlo >> s) & 1u) {
              tc_mma_bf16(tmem, a, b, idesc, 1u);
              tc_mma_bf16(tmem, a + 2, b + 2, idesc, 1u);
            }
            if (BK == 64 && ((whi >> s) & 1u)) {
              tc_mma_bf16(tmem, a + 4, b + 4, idesc, 1u);
              tc_mma_bf16(tmem, a + 6, b + 6, idesc, 1u);
            }
            tc_commit(bar_empty + 8 * s);
          }
        }
        __syncwarp();
        a += L::kStage / 16;
        b += L::kStage / 16;
      }
      ph = 1u;
      // the listed ones, unrolled again: bit s of mlo, mhi: the first, last 32
      // columns of stage s take part (a convolution's listed blocks are whole)
      uint32_t mlo = 0xFFu, mhi = 0xFFu;
      for (int i0 = kStages; ok && i0 < total; i0 += kStages) {
        if (p.conv == 0) {
          bool flo = false, fhi = false;
          if (lane < kStages && i0 + lane < total) {
            const int kb = listed_block(i0 - kStages + lane);
            flo = ((s_lo[kb >> 5] >> (kb & 31)) & 1u) != 0u;
            fhi = BK == 32 || ((s_hi[kb >> 5] >> (kb & 31)) & 1u) != 0u;
          }
          mlo = __ballot_sync(0xffffffffu, flo);
          mhi = __ballot_sync(0xffffffffu, fhi);
        }
#pragma unroll
        for (int s = 0; s < kStages; ++s) {
          if (ok && i0 + s < total) {
            ok = mbar_wait_warp(bar_full + 8 * s, ph, err, s_abort, kErrTimeoutFull, wlim);
            if (ok) {
              tc_fence_after();
              const uint64_t as = ad + (uint64_t)(s * (L::kStage / 16)), bs = bd + (uint64_t)(s * (L::kStage / 16));
              if (((mlo & mhi) >> s) & 1u) {
                if (el) {
#pragma unroll
                  for (int k = 0; k < BK / 16; ++k)
                    tc_mma_bf16(tmem, as + (uint64_t)(2 * k), bs + (uint64_t)(2 * k), idesc, 1u);
                  tc_commit(bar_empty + 8 * s);
                }
              } else if (el) {  // one half
                const uint64_t k0 = ((mlo >> s) & 1u) ? 0u : 4u;
                tc_mma_bf16(tmem, as + k0, bs + k0, idesc, 1u);
                tc_mma_bf16(tmem, as + k0 + 2, bs + k0 + 2, idesc, 1u);
                tc_commit(bar_empty + 8 * s);
              }
            }
            __syncwarp();
          }
        }
        ph ^= 1u;
      }
    }
    // (the error-path tests leave the accumulator unsignalled)
    if (ok && el && P.fault != kFaultSkipFirstAccCommit) tc_commit(bar_acc);
    __syncwarp();
    cluster_arrive();
    cluster_wait();
  } else {
    // ------------------------------------------------------------------ producers
    if (listed) named_bar_sync(2, kThreads);
    const int rest = listed ? listed_rest() : span - lap;
    if (lane == 0) {
      int fills = warp < lap ? 1 : 0;
      for (int i = warp; i < rest; i += kStages, ++fills) {  // (only when lap == kStages)
        if (!mbar_wait(bar_empty + 8 * warp, (uint32_t)((fills - 1) & 1), err, s_abort, kErrTimeoutEmpty, wlim)) break;
        const int kb = kb0 + (listed ? listed_block(i) : kStages + i);
        mbar_arrive_expect_tx(fb, stage_bytes);
        load_b(kb);
        seek_a(kb);
        load_a();
      }
      s_issued[warp] = fills;
    }
    __syncwarp();
    // ------------------------------------------------------------------ epilogue
    float sc[4] = {1.f, 1.f, 1.f, 1.f}, sh[4] = {0.f, 0.f, 0.f, 0.f};
    if (cvalid)
#pragma unroll
      for (int i = 0; i < 4; ++i) epi_affine(P.ep, p.N, col + i, sc[i], sh[i]);
    uint2 res[kIters];
#pragma unroll
    for (int i = 0; i < kIters; ++i) {
      res[i] = make_uint2(0u, 0u);
      if (P.ep.residual && mrow[i] >= 0)
        res[i] = *reinterpret_cast<const uint2*>(P.ep.residual + (int64_t)mrow[i] * p.N + col);
    }
    const uint32_t part = sbase;  // [128][kPitch] fp32, in the ring's memory
    bool ok = mbar_wait_spin(bar_acc, 0u, err, s_abort, kErrTimeoutAcc, wlim);
    ok = !named_bar_or(1, kWorkers, !ok);
    if (ok) {
      const int q = warp & 3, hf = warp >> 2;
      const uint32_t dst = part + (uint32_t)((q * 32 + lane) * kPitch + hf * 32) * 4;
      uint32_t raw[32];
      tc_fence_after();
      tmem_ld32_nowait(tmem + ((uint32_t)(q * 32) << 16) + (uint32_t)(hf * 32), raw);
      tmem_wait_ld32(raw);
      tc_fence_before();
#pragma unroll
      for (int i = 0; i < 8; ++i)
        sts_u4(dst + 16 * i, make_uint4(raw[4 * i], raw[4 * i + 1], raw[4 * i + 2], raw[4 * i + 3]));
    }
    cluster_arrive();
    cluster_wait();
    if (ok) {
      const OccDev o = P.out_occ;
      const int emit = P.emit;
      const int act = P.ep.act;
      // the shares' partial sums of this thread's values, all loads in flight
      float4 w[kIters][KS];
#pragma unroll
      for (int i = 0; i < kIters; ++i) {
        const uint32_t src =
            part + (uint32_t)(((i * 16 + ((int)threadIdx.x >> 4)) * KS + rank) * kPitch + 4 * c4) * 4;
#pragma unroll
        for (int k = 0; k < KS; ++k) {
          w[i][k] = make_float4(0.f, 0.f, 0.f, 0.f);
          if (mrow[i] >= 0) w[i][k] = ld_cluster_f4(cluster_map(src, (uint32_t)k));
        }
      }
      uint32_t cnt[4] = {0u, 0u, 0u, 0u};
#pragma unroll
      for (int i = 0; i < kIters; ++i) {
        float4 v = w[i][0];
#pragma unroll
        for (int k = 1; k < KS; ++k) {  // in rank order
          v.x += w[i][k].x;
          v.y += w[i][k].y;
          v.z += w[i][k].z;
          v.w += w[i][k].w;
        }
        const bool live = mrow[i] >= 0;
        const int64_t m = mrow[i];
        v.x = fmaf(v.x, sc[0], sh[0]);
        v.y = fmaf(v.y, sc[1], sh[1]);
        v.z = fmaf(v.z, sc[2], sh[2]);
        v.w = fmaf(v.w, sc[3], sh[3]);
        if (P.ep.residual) {
          v.x += __uint_as_float(res[i].x << 16);
          v.y += __uint_as_float(res[i].x & 0xFFFF0000u);
          v.z += __uint_as_float(res[i].y << 16);
          v.w += __uint_as_float(res[i].y & 0xFFFF0000u);
        }
        if (P.y_f32) {
          if (live)
            *reinterpret_cast<float4*>(static_cast<float*>(P.y) + m * p.N + col) =
                make_float4(epi_act(v.x, act), epi_act(v.y, act), epi_act(v.z, act), epi_act(v.w, act));
          continue;
        }
        uint2 pk;
        if (act == 1) {
          pk.x = act_pack2<1>(v.x, v.y);
          pk.y = act_pack2<1>(v.z, v.w);
        } else if (act == 2) {
          pk.x = act_pack2<2>(v.x, v.y);
          pk.y = act_pack2<2>(v.z, v.w);
        } else if (act == 0) {
          pk.x = act_pack2<0>(v.x, v.y);
          pk.y = act_pack2<0>(v.z, v.w);
        } else {
          pk.x = act_pack2<3>(v.x, v.y);
          pk.y = act_pack2<3>(v.z, v.w);
        }
        if (live) *reinterpret_cast<uint2*>(static_cast<__nv_bfloat16*>(P.y) + m * p.N + col) = pk;
        if (emit) {
          uint32_t nib = 0u;
          if (live) {
            const uint32_t nx = nz_pairs(pk.x), ny = nz_pairs(pk.y);
            cnt[0] += nx & 1u;
            cnt[1] += nx >> 16;
            cnt[2] += ny & 1u;
            cnt[3] += ny >> 16;
            nib = (nx | (nx >> 15) | (ny << 2) | (ny >> 13)) & 15u;
          }
          uint32_t word = nib << (4 * (lane & 7));
          word |= __shfl_xor_sync(0xffffffffu, word, 1);
          word |= __shfl_xor_sync(0xffffffffu, word, 2);
          word |= __shfl_xor_sync(0xffffffffu, word, 4);
          if ((lane & 7) == 0) s_word[(i * 16 + ((int)threadIdx.x >> 4)) * 2 + (c4 >> 3)] = word;
        }
      }
      if (emit) {
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          cnt[i] += __shfl_xor_sync(0xffffffffu, cnt[i], 16);
          if (lane < 16 && cnt[i]) atomicAdd(&s_cnt[4 * c4 + i], cnt[i]);
        }
        named_bar_sync(1, kWorkers);
        if (threadIdx.x < 2 * kRows) {
          // thread = one 32-column word of one row; the words of a warp that
          // belong to the same 128-row block leave as one atomic
          const int row = (int)threadIdx.x >> 1;
          bool v;
          int img, oh, ow;
          const int64_t m = tile_row(p, g, row * KS + rank, v, img, oh, ow);
          const uint32_t word = s_word[threadIdx.x];
          const bool row_nz = (word | __shfl_xor_sync(0xffffffffu, word, 1)) != 0u;
          if ((lane & 1) == 0 && row_nz) {
            unsigned long long* dst = &o.row_bm[m * o.W64 + (g.n0 >> 12)];
            const unsigned long long bit = 1ull << ((g.n0 >> 6) & 63);
            if (nt == 1) *dst = bit;
            else atomicOr(dst, bit);
          }
          const int key = word ? (int)(m >> 7) * o.C32 + (g.n0 >> 5) + (lane & 1) : -1;
          const uint32_t same = __match_any_sync(0xffffffffu, key);
          const uint32_t bits = __reduce_or_sync(same, word);
          if (key >= 0 && (int)__ffs(same) - 1 == lane) atomicOr(&o.blk_mask[key], bits);
        }
        if (threadIdx.x < kBN) {
          const uint32_t c = s_cnt[threadIdx.x];
          const uint32_t sum = __reduce_add_sync(0xffffffffu, c);
          if (c) atomicAdd(&o.col_nnz[g.n0 + threadIdx.x], c);  // (columns past N have none)
          if (lane == 0 && sum) {
            atomicAdd(&o.tile_nnz[g.n0 >> 6], sum);
            atomicAdd(o.nnz, (unsigned long long)sum);
          }
        }
      }
    }
  }
  // no CTA of the cluster leaves while another may read its partial tile
  // (every value read has been used: no ordering of memory is needed)
  __syncwarp();
  if (KS > 1) {
    cluster_arrive_relaxed();
    cluster_wait();
  }
  if (*s_abort) {
    // a bounded wait ran out: the copies and MMAs issued so far finish
    // (bounded again) before shared and tensor memory are released
    if (warp < kWarps && lane == 0 && s_issued[warp] > 0)
      mbar_drain(fb, (uint32_t)((s_issued[warp] - 1) & 1), wlim);
    if (warp == kWarps && elect_one()) {
      tc_commit(bar_drain);
      mbar_drain(bar_drain, 0u, wlim);
    }
    __syncwarp();
  }
  tc_fence_before();
  __syncthreads();
  if (warp == kWarps) {
    tc_fence_after();
    tmem_dealloc(tmem, kTmemCols);
  }
}

template <int BK, int KS>
cudaError_t launch_ks(const IgemmArgs& a, const CUtensorMap& tA, const CUtensorMap& tB, int64_t tiles, int a_rows,
                      cudaStream_t s) {
  const void* f = reinterpret_cast<const void*>(onetile_kernel<BK, KS>);
  const cudaError_t e0 = smem_optin(f, (size_t)Lay<BK>::kSmem);
  if (e0 != cudaSuccess) return e0;
  const cudaError_t e = launch_cluster_kernel(onetile_kernel<BK, KS>, dim3((unsigned)(tiles * KS)), dim3(kThreads),
                                              (unsigned)KS, (size_t)Lay<BK>::kSmem, s, tA, tB, a, a_rows);
  if (e != cudaSuccess) return e;
  return cudaGetLastError();
}

template <int BK>
cudaError_t launch_bk(const IgemmArgs& a, const CUtensorMap& tA, const CUtensorMap& tB, int64_t tiles, int a_rows,
                      cudaStream_t s) {
  switch (a.ksplit) {
    case 1: return launch_ks<BK, 1>(a, tA, tB, tiles, a_rows, s);
    case 2: return launch_ks<BK, 2>(a, tA, tB, tiles, a_rows, s);
    case 4: return launch_ks<BK, 4>(a, tA, tB, tiles, a_rows, s);
    default: return launch_ks<BK, 8>(a, tA, tB, tiles, a_rows, s);
  }
}

}  // namespace

// Clusters of `ks` CTAs that the device runs at once, asked once per device: a
// cluster lies within one GPC and a CTA fills an SM, so 152 SMs hold 15 clusters
// of 8 and 36 of 4 (a second round doubles the time: 128 x 1024 x 512, 16 tiles,
// by 8 8.4 us, by 4 4.3 us).
namespace {
int clusters_at_once(int ks) {
  constexpr int kDevices = 64;
  static std::mutex mu;
  static int known[kDevices][4];  // 0: not asked yet
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return 0;
  const int at = ks == 8 ? 3 : ks == 4 ? 2 : ks == 2 ? 1 : 0;
  std::lock_guard<std::mutex> lock(mu);
  if (dev < kDevices && known[dev][at] > 0) return known[dev][at];
  const void* f = ks == 8   ? reinterpret_cast<const void*>(onetile_kernel<64, 8>)
                  : ks == 4 ? reinterpret_cast<const void*>(onetile_kernel<64, 4>)
                  : ks == 2 ? reinterpret_cast<const void*>(onetile_kernel<64, 2>)
                            : reinterpret_cast<const void*>(onetile_kernel<64, 1>);
  if (smem_optin(f, (size_t)Lay<64>::kSmem) != cudaSuccess) return 0;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)ks);
  cfg.blockDim = dim3(kThreads);
  cfg.dynamicSmemBytes = (size_t)Lay<64>::kSmem;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = (unsigned)ks;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  int n = 0;
  if (cudaOccupancyMaxActiveClusters(&n, f, &cfg) != cudaSuccess) {
    cudaGetLastError();  // (not the launch's error)
    return 0;
  }
  if (dev < kDevices) known[dev][at] = n;
  return n;
}
}  // namespace

// Cluster size: the largest of 8, 4 and 2 whose clusters all run at once and whose
// CTAs keep enough K blocks, 1 for long K; else the persistent kernel.  On 128 rows,
// dense, without / with occupancy (and its clear), us:
//   K = 64     77 tiles            by 1 5.1 / 7.8   persistent 3.8 / 6.4
//   K = 256    24 tiles, by 4 4.5 / 6.3             4.3 / 6.9
//   K = 512    24 tiles, by 4 4.9 / 6.9             5.1 / 7.7
//              76 tiles, by 2 6.0 / 8.5             5.3 / 7.9
//   K = 768    76 tiles, by 2 6.2 / 8.7             6.0 / 8.6
//   K = 1152   14 tiles, by 8 5.0 / 6.8, by 4 4.7 / 6.8
//              90 tiles            by 1 8.6 / 11.1  7.4 / 10.0
//   K = 4608   90 tiles            by 1 18.2 / 21.1  19.8 / 22.6
// A convolution's zero-skip path is much slower in the persistent kernel (its
// masks, then its loads, tile by tile: [8,28,28,128] 3x3 by 1 13, persistent 19.6;
// dense 11.4 and 11.2), so unless the dense path is forced it takes what fits.
// fp32 output (`lean` false), whose persistent kernel is slower, takes what fits.
int onetile_split(const IgemmArgs& a, int64_t mtiles, int bk, bool lean) {
  const int64_t tiles = mtiles * ((a.N + kBN - 1) / kBN);
  const int kblocks = (a.Ktot + bk - 1) / bk;
  if (a.conv == 1 || tiles > device_sm_count() || kblocks > kMaxItems) return 0;
  for (int ks = 8; ks >= 1; ks /= 2) {
    const int least = !lean        ? ks
                      : ks == 8    ? 24
                      : a.conv && a.disp.force != 1 ? ks
                      : ks == 4    ? (a.emit ? 4 : 8)
                      : ks == 2    ? (a.emit ? 8 : 12)
                                   : 48;
    if (kblocks >= least && tiles * ks <= device_sm_count() && (ks == 1 || tiles <= clusters_at_once(ks))) return ks;
  }
  return 0;
}

cudaError_t launch_onetile(const IgemmArgs& a, int64_t mtiles, int bk, cudaStream_t s) {
  CUtensorMap tA, tB;
  int a_rows = kBM;
  if (a.conv == 0) {
    a_rows = a.M < kBM ? a.M : kBM;
    if (!make_tmap_2d(&tA, a.x, (uint64_t)a.M, (uint64_t)a.Ktot, (uint32_t)bk, (uint32_t)a_rows))
      return cudaErrorInvalidValue;
  } else {
    const int bn = a.bn < a.Nimg ? a.bn : a.Nimg;
    a_rows = a.bw * a.bh * bn;
    if (!make_tmap_nhwc(&tA, a.x, a.Nimg, a.H, a.W, a.Cp, bk, a.bw, a.bh, bn, a.stride))
      return cudaErrorInvalidValue;
  }
  if (!make_tmap_2d(&tB, a.w, (uint64_t)a.N, (uint64_t)a.Ktot, (uint32_t)bk, kBN)) return cudaErrorInvalidValue;
  const int64_t tiles = mtiles * ((a.N + kBN - 1) / kBN);
  return bk == 64 ? launch_bk<64>(a, tA, tB, tiles, a_rows, s) : launch_bk<32>(a, tA, tB, tiles, a_rows, s);
}

}  // namespace sparoa
